// Set operations of the HOLD integrator (Appendix A): gathers of a set's
// bodies into compact arrays, the stable split of a set into slow and fast
// bodies, kicks and drifts of a set. The recursion over large sets and
// their force solves are driven from the host (api.cu, fmm_hold); a small set
// evolves entirely inside one block (k_hold_small), recursion included.
//
// Compiled with -fmad=false: a drift x + dt v and a kick v + h a round as
// two operations, as the oracle does.
#include "gbfmm_internal.cuh"
#include "hold_bounds.cuh"
#include "hold_pair.cuh"

namespace gbfmm {

namespace {

inline int grid_for(int64_t n, int threads) { return (int)((n + threads - 1) / threads); }

// out[c][a] = field c of body idx[a]: x, y, z, vx, vy, vz, m (7 arrays of k);
// zero_from >= 0 zeroes the masses of a >= zero_from
__global__ void k_hold_gather(int k, const int* __restrict__ idx, const double* __restrict__ x,
                              const double* __restrict__ y, const double* __restrict__ z,
                              const double* __restrict__ vx, const double* __restrict__ vy,
                              const double* __restrict__ vz, const double* __restrict__ m, double* __restrict__ out,
                              int stride, int zero_from) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= k) return;
    const int i = idx[a];
    out[a] = x[i];
    out[stride + a] = y[i];
    out[2 * (size_t)stride + a] = z[i];
    out[3 * (size_t)stride + a] = vx[i];
    out[4 * (size_t)stride + a] = vy[i];
    out[5 * (size_t)stride + a] = vz[i];
    out[6 * (size_t)stride + a] = (zero_from >= 0 && a >= zero_from) ? 0.0 : m[i];
}

__global__ void k_hold_flags(int k, const double* __restrict__ tau, double dt, uint32_t* __restrict__ flag) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a < k) flag[a] = tau[a] < dt ? 1u : 0u;
}

// stable split by an exclusive scan of the fast flags
__global__ void k_hold_compact(int k, const int* __restrict__ idx, const uint32_t* __restrict__ flag,
                               const uint32_t* __restrict__ scan, int* __restrict__ S, int* __restrict__ F) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= k) return;
    const uint32_t f = scan[a];
    if (flag[a]) F[f] = idx[a];
    else S[a - f] = idx[a];
}

// v[idx[a]] += h (acc[a] - sub[a]) (sub may be NULL); acc: 3 arrays of stride
__global__ void k_hold_kick(int k, const int* __restrict__ idx, const double* __restrict__ acc,
                            const double* __restrict__ sub, int stride, int sub_stride, double h,
                            double* __restrict__ vx, double* __restrict__ vy, double* __restrict__ vz) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= k) return;
    const int i = idx[a];
    double ax = acc[a], ay = acc[stride + a], az = acc[2 * (size_t)stride + a];
    if (sub) {
        ax = ax - sub[a];
        ay = ay - sub[sub_stride + a];
        az = az - sub[2 * (size_t)sub_stride + a];
    }
    vx[i] = vx[i] + h * ax;
    vy[i] = vy[i] + h * ay;
    vz[i] = vz[i] + h * az;
}

__global__ void k_hold_drift(int k, const int* __restrict__ idx, double dt, double* __restrict__ x,
                             double* __restrict__ y, double* __restrict__ z, const double* __restrict__ vx,
                             const double* __restrict__ vy, const double* __restrict__ vz) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= k) return;
    const int i = idx[a];
    x[i] = x[i] + dt * vx[i];
    y[i] = y[i] + dt * vy[i];
    z[i] = z[i] + dt * vz[i];
}

__global__ void k_hold_iota(int n, int* __restrict__ idx) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a < n) idx[a] = a;
}

// ---------------------------------------------------------------------------
// Device-resident HOLD for a small set: evolve(P, dt) of Appendix A for the k
// bodies idx[0..k), recursion included, in one block. The set's positions,
// velocities and masses are copied into shared memory; every subset of the
// recursion is a segment of the index array ix, split in place (stable: slow
// bodies first, then fast ones). A frame's split is kept as a bit mask and
// undone when the frame ends, so the parent sees its fast set in its own
// order again, as the oracle (fresh S and F arrays per level) does. Forces
// are the oracle's FP64 direct sum in the oracle's order and operations
// (r = sqrt(r^2), m / (r^2 r), no contraction), and a body is fast when the same
// tau_pair says so: the trajectory is the oracle's bit for bit.
//
// One SM's FP64 pipe (two lanes a clock) bounds it, and the latency of the
// steps in the small sets deep in the recursion. So
//  - the split needs only to know whether some pair step is below dt: FP32
//    bounds (hold_bounds.cuh) decide nearly every pair, the rest are evaluated
//    exactly;
//  - a kick runs over the unordered pairs with a slow member, one thread each:
//    r and r^3 serve both bodies, whose two terms go to shared memory, and one
//    thread per body and component adds its terms in source order.
// N = 100 (a Plummer sphere, dt = 1/16, one step): 30.1 -> 4.1 ms against one thread
// per body, every pair step exact and every force pair from both sides.

struct HoldFrame {
    double dt;
    int lo, hi;   // the set: ix[lo..hi)
    int ns;       // slow bodies ix[lo..lo+ns) after the split; fast ones after them
    int phase;    // 0: split and evolve the fast set; 1: kick-drift-kick, fast again; 2: undo the split
    int depth;
    int pad;
};

constexpr int kHoldThreads = 256;

constexpr int kHoldPairs = 1024;  // pairs whose terms are in shared memory at a time (>= kHoldSmallMax)
constexpr int kHoldWhole = kHoldPairs / 4;  // sets up to here always have four whole rows in a chunk
constexpr int kHoldRows = 16;               // rows of a chunk of a larger set's pairs
constexpr int kHoldUnsure = 256;  // pairs the bounds leave open, listed before they are evaluated

// shared memory of a kick's terms or a split's FP32 members
__host__ __device__ constexpr size_t hold_term_bytes(int k) {
    return 6 * kHoldPairs * sizeof(double) > (size_t)k * sizeof(PairBody32) ? 6 * kHoldPairs * sizeof(double)
                                                                           : (size_t)k * sizeof(PairBody32);
}

// The two terms of pair (a, b) of a set, on a and on b, to term[e].
__device__ __forceinline__ void kick_pair(const int* ix, int a, int b, const double* px, const double* py,
                                          const double* pz, const double* pm, double soft2, double* term, int e) {
    const int i = ix[a], j = ix[b];
    const double dx = px[j] - px[i], dy = py[j] - py[i], dz = pz[j] - pz[i];
    double r2 = dx * dx + dy * dy + dz * dz;
    if (soft2 > 0.0) r2 = r2 + soft2;
    const double r = sqrt(r2);
    const double r3 = r2 * r;
    const double ma = pm[j] / r3, mb = pm[i] / r3;
    term[e] = ma * dx;
    term[kHoldPairs + e] = ma * dy;
    term[2 * kHoldPairs + e] = ma * dz;
    // (the pair seen from b: exactly the opposite offsets)
    term[3 * kHoldPairs + e] = mb * -dx;
    term[4 * kHoldPairs + e] = mb * -dy;
    term[5 * kHoldPairs + e] = mb * -dz;
}

// The sums of a kick where few rows of a set fit in term: chunks of kHoldRows rows,
// each in tiles of columns from the chunk's first row on. A body's column comes in the
// chunks of the rows below it, then its row with the columns above it, tile by tile.
__device__ void kick_sums_tiled(const int* ix, int n, int ns, const double* px, const double* py,
                                             const double* pz, const double* pm, double soft2, double* acc,
                                             double* term) {
    const int tid = threadIdx.x;
    const int rows = kHoldRows < ns ? kHoldRows : ns, cols = kHoldPairs / rows;  // (cols >= rows)
    for (int a0 = 0; a0 < ns; a0 += rows) {
        const int a1 = a0 + rows < ns ? a0 + rows : ns;
        for (int c0 = a0; c0 < n; c0 += cols) {
            const int c1 = c0 + cols < n ? c0 + cols : n, w = c1 - c0;
            for (int e = tid; e < (a1 - a0) * w; e += kHoldThreads) {
                const int a = a0 + e / w, b = c0 + e % w;
                if (b > a) kick_pair(ix, a, b, px, py, pz, pm, soft2, term, e);
            }
            __syncthreads();
            // the columns' sums and, after the first tile, where they are no longer columns, the rows'
            const int ncol = 3 * w, nrow = c0 > a0 ? 3 * (a1 - a0) : 0;
            for (int e = tid; e < ncol + nrow; e += kHoldThreads) {
                const int c = e % 3, s = e < ncol ? c0 + e / 3 : a0 + (e - ncol) / 3;
                const double* on_b = term + (3 + c) * kHoldPairs + (s - c0);
                const double* on_a = term + c * kHoldPairs + (s - a0) * w - c0;
                double v = acc[3 * s + c];
                if (e < ncol)
                    for (int a = a0; a < a1 && a < s; ++a) v += on_b[(a - a0) * w];
                if (s < a1)
                    for (int b = s + 1 > c0 ? s + 1 : c0; b < c1; ++b) v += on_a[b];
                acc[3 * s + c] = v;
            }
            __syncthreads();
        }
    }
}

// Kick of the set ix[0..n), its first ns members slow: slow bodies feel
// all of it, fast ones the slow ones; v <- v + h G sum, sources in set order,
// a body not acting on itself. Rows a = 0..ns-1 of pairs (a, b), a < b, in
// chunks: a chunk holds for each of its rows the pairs with every b > a, so a
// body s adds its sources in order: those of the chunk's rows below s, then,
// if s is itself a row of the chunk, those above s. acc: 3 n sums; term:
// 6 kHoldPairs values (on a from b, then on b from a).
//
// A row's sum is serial, and an FP64 instruction takes the pipe as long for one lane as
// for 32, so a chunk needs several rows: where fewer than four (and not all) fit, rows
// come in tiles (LARGE; in a kernel of their own, as the code costs the small sets 1 to 4 %). Kicks of a whole set, ms each, one thread per body | whole rows |
// tiles: 256 bodies 1.7 | 0.9 | -, 512 7.0 | 4.7 | 2.2, 700 13.1 | 13.6 | 4.0, 1024 27.9 | 28.4 | 8.6.
template <bool LARGE>
__device__ void set_kick(const int* ix, int n, int ns, const double* px, const double* py, const double* pz,
                          const double* pm, double* pvx, double* pvy, double* pvz, double G, double soft2, double h,
                          double* acc, double* term) {
    const int tid = threadIdx.x;
    const int fit = kHoldPairs / n, rows = fit < ns ? fit : ns;
    for (int e = tid; e < 3 * n; e += kHoldThreads) acc[e] = 0.0;
    if (LARGE && fit < 4 && fit < ns) {
        kick_sums_tiled(ix, n, ns, px, py, pz, pm, soft2, acc, term);
    } else {
        for (int a0 = 0; a0 < ns; a0 += rows) {
            const int a1 = a0 + rows < ns ? a0 + rows : ns;
            for (int e = tid; e < (a1 - a0) * n; e += kHoldThreads) {
                const int a = a0 + e / n, b = e % n;
                if (b > a) kick_pair(ix, a, b, px, py, pz, pm, soft2, term, e);
            }
            __syncthreads();
            for (int e = a0 * 3 + tid; e < 3 * n; e += kHoldThreads) {  // bodies below a0 have all their sources
                const int s = e / 3, c = e - 3 * s;
                const double* on_b = term + (3 + c) * kHoldPairs + s;
                const double* on_a = term + c * kHoldPairs + (s - a0) * n;
                double v = acc[e];
                for (int a = a0; a < a1 && a < s; ++a) v += on_b[(a - a0) * n];
                if (s < a1)
                    for (int b = s + 1; b < n; ++b) v += on_a[b];
                acc[e] = v;
            }
            __syncthreads();
        }
    }
    for (int s = tid; s < n; s += kHoldThreads) {
        const int i = ix[s];
        pvx[i] += h * (G * acc[3 * s]);
        pvy[i] += h * (G * acc[3 * s + 1]);
        pvz[i] += h * (G * acc[3 * s + 2]);
    }
    __syncthreads();
}

// The fast members of the set ix[0..n) as bits: those with a pair step below
// dt. b32: the members in FP32 pairs (scratch), unsure: kHoldUnsure words.
__device__ void set_fast_bits(const int* ix, int n, const double* px, const double* py, const double* pz,
                               const double* pvx, const double* pvy, const double* pvz, const double* pm, double G,
                               double eta, bool sym, double dt, PairBody32* b32, unsigned* bits, unsigned* unsure,
                               int* nunsure) {
    const int tid = threadIdx.x;
    for (int t = tid; t < n; t += kHoldThreads) {
        const int i = ix[t];
        b32[t] = PairBody32(px[i], py[i], pz[i], pvx[i], pvy[i], pvz[i], pm[i]);
    }
    if (tid < ((n + 31) >> 5)) bits[tid] = 0u;
    if (tid == 0) *nunsure = 0;
    __syncthreads();
    const float dtf = (float)dt;  // its rounding is far inside the bounds' margin
    auto mark = [&](int a, int b) {
        atomicOr(bits + (a >> 5), 1u << (a & 31));
        atomicOr(bits + (b >> 5), 1u << (b & 31));
    };
    auto exact = [&](int a, int b) {
        const int i = ix[a], j = ix[b];
        if (tau_pair(px[j] - px[i], py[j] - py[i], pz[j] - pz[i], pvx[j] - pvx[i], pvy[j] - pvy[i], pvz[j] - pvz[i],
                     pm[i] + pm[j], G, eta, sym) < dt)
            mark(a, b);
    };
    const int np = n * (n - 1) / 2;
    for (int p = tid; p < np; p += kHoldThreads) {
        int b = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)p)) * 0.5f);  // p = b (b - 1) / 2 + a, a < b
        while (b * (b - 1) / 2 > p) --b;
        while (b * (b + 1) / 2 <= p) ++b;
        const int a = p - b * (b - 1) / 2;
        const PairScale32 scale(b32[a], G, eta);
        float lo, hi;
        // (equal velocities are rare after a first kick: such a pair is evaluated)
        pair_bounds32(b32[a], b32[b], scale, sym, [] { return false; }, lo, hi);
        if (hi < dtf) {
            mark(a, b);
        } else if (lo < dtf) {
            const int k = atomicAdd(nunsure, 1);
            if (k < kHoldUnsure) unsure[k] = (unsigned)a << 16 | (unsigned)b;
            else exact(a, b);
        }
    }
    __syncthreads();
    const int nu = *nunsure < kHoldUnsure ? *nunsure : kHoldUnsure;
    for (int k = tid; k < nu; k += kHoldThreads) {
        const int a = (int)(unsure[k] >> 16), b = (int)(unsure[k] & 0xffffu);
        // (a bit set meanwhile by another pair only saves the evaluation)
        const unsigned wa = *(volatile unsigned*)(bits + (a >> 5)), wb = *(volatile unsigned*)(bits + (b >> 5));
        if (!((wa >> (a & 31)) & (wb >> (b & 31)) & 1u)) exact(a, b);
    }
    __syncthreads();
}

// stats: {slow-system kicks, FMM solves (none here), direct solves, deepest level, splits}
// LARGE: k may be above kHoldWhole
template <bool LARGE>
__global__ void __launch_bounds__(kHoldThreads) k_hold_small(int k, const int* __restrict__ idx, double* x,
                                                             double* y, double* z, double* vx, double* vy,
                                                             double* vz, const double* __restrict__ m, double G,
                                                             double soft2, double eta, int sym, double dt,
                                                             double dt_min, int depth0,
                                                             unsigned long long* __restrict__ stats) {
    extern __shared__ __align__(16) double hsm[];
    const int W = (k + 31) >> 5;  // mask words per level
    double* px = hsm;
    double* py = px + k;
    double* pz = py + k;
    double* pvx = pz + k;
    double* pvy = pvx + k;
    double* pvz = pvy + k;
    double* pm = pvz + k;
    double* acc = pm + k;                                      // 3 k sums of a kick
    double* term = acc + 3 * k;                                // its pairs' terms
    HoldFrame* stack = reinterpret_cast<HoldFrame*>(reinterpret_cast<unsigned char*>(term) + hold_term_bytes(k));
    int* ix = reinterpret_cast<int*>(stack + kHoldMaxLevels);
    int* tmp = ix + k;
    unsigned* fbits = reinterpret_cast<unsigned*>(tmp + k);  // kHoldMaxLevels x W
    // the members in FP32 pairs share the terms' memory (a split and a kick never overlap)
    PairBody32* b32 = reinterpret_cast<PairBody32*>(term);
    __shared__ unsigned s_unsure[kHoldUnsure];
    __shared__ int s_sp, s_nf, s_nunsure;
    const int tid = threadIdx.x;
    for (int a = tid; a < k; a += kHoldThreads) {
        const int i = idx[a];
        px[a] = x[i]; py[a] = y[i]; pz[a] = z[i];
        pvx[a] = vx[i]; pvy[a] = vy[i]; pvz[a] = vz[i];
        pm[a] = m[i];
        ix[a] = a;
    }
    unsigned long long kicks = 0, direct = 0, splits = 0, deepest = 0;
    if (tid == 0) {
        stack[0] = HoldFrame{dt, 0, k, k, 0, depth0, 0};
        s_sp = 0;
    }
    __syncthreads();
    for (;;) {
        const int sp = s_sp;
        if (sp < 0) break;
        const HoldFrame f = stack[sp];
        __syncthreads();  // every thread has its copy before thread 0 edits the stack
        const int n = f.hi - f.lo;
        unsigned* bits = fbits + (size_t)sp * W;
        if (f.phase == 0) {
            if ((unsigned long long)f.depth > deepest) deepest = (unsigned long long)f.depth;
            int ns = n;
            if (n > 1 && f.dt > dt_min && f.depth < kHoldMaxDepth && sp + 1 < kHoldMaxLevels) {
                set_fast_bits(ix + f.lo, n, px, py, pz, pvx, pvy, pvz, pm, G, eta, sym != 0, f.dt, b32, bits,
                               s_unsure, &s_nunsure);
                if (tid == 0) s_nf = 0;
                __syncthreads();
                if (tid < ((n + 31) >> 5)) atomicAdd(&s_nf, __popc(bits[tid]));
                __syncthreads();
                const int nf = s_nf;
                ns = n - nf;
                // stable split into tmp, back into the segment
                for (int t = tid; t < n; t += kHoldThreads) {
                    int before = 0;
                    for (int w = 0; w < (t >> 5); ++w) before += __popc(bits[w]);
                    const unsigned word = bits[t >> 5];
                    before += __popc(word & ((1u << (t & 31)) - 1u));
                    const bool fast = (word >> (t & 31)) & 1u;
                    tmp[fast ? ns + before : t - before] = ix[f.lo + t];
                }
                __syncthreads();
                for (int t = tid; t < n; t += kHoldThreads) ix[f.lo + t] = tmp[t];
                ++splits;
            }
            if (tid == 0) {
                stack[sp].ns = ns;
                stack[sp].phase = 1;
                if (ns < n) {
                    stack[sp + 1] = HoldFrame{0.5 * f.dt, f.lo + ns, f.hi, f.hi - f.lo - ns, 0, f.depth + 1, 0};
                    s_sp = sp + 1;
                }
            }
            __syncthreads();
            continue;
        }
        if (f.phase == 1) {
            const int s1 = f.lo + f.ns;
            if (f.ns > 0) {
                // slow bodies feel all of P, fast ones the slow ones; drift the slow ones
                const double h = 0.5 * f.dt;
                set_kick<LARGE>(ix + f.lo, n, f.ns, px, py, pz, pm, pvx, pvy, pvz, G, soft2, h, acc, term);
                for (int t = f.lo + tid; t < s1; t += kHoldThreads) {
                    const int i = ix[t];
                    px[i] += f.dt * pvx[i];
                    py[i] += f.dt * pvy[i];
                    pz[i] += f.dt * pvz[i];
                }
                __syncthreads();
                set_kick<LARGE>(ix + f.lo, n, f.ns, px, py, pz, pm, pvx, pvy, pvz, G, soft2, h, acc, term);
                kicks += 2;
                direct += (f.ns < n) ? 4 : 2;
            }
            __syncthreads();
            if (tid == 0) {
                stack[sp].phase = 2;
                if (f.ns < n) {
                    stack[sp + 1] = HoldFrame{0.5 * f.dt, s1, f.hi, f.hi - s1, 0, f.depth + 1, 0};
                    s_sp = sp + 1;
                }
            }
            __syncthreads();
            continue;
        }
        // phase 2: undo this frame's split (its children undid theirs), then return
        if (f.ns < n) {
            for (int t = tid; t < n; t += kHoldThreads) {
                int before = 0;
                for (int w = 0; w < (t >> 5); ++w) before += __popc(bits[w]);
                const unsigned word = bits[t >> 5];
                before += __popc(word & ((1u << (t & 31)) - 1u));
                const bool fast = (word >> (t & 31)) & 1u;
                tmp[t] = ix[f.lo + (fast ? f.ns + before : t - before)];
            }
            __syncthreads();
            for (int t = tid; t < n; t += kHoldThreads) ix[f.lo + t] = tmp[t];
        }
        if (tid == 0) s_sp = sp - 1;
        __syncthreads();
    }
    for (int a = tid; a < k; a += kHoldThreads) {
        const int i = idx[a];
        x[i] = px[a]; y[i] = py[a]; z[i] = pz[a];
        vx[i] = pvx[a]; vy[i] = pvy[a]; vz[i] = pvz[a];
    }
    if (tid == 0) {
        atomicAdd(stats + 0, kicks);
        atomicAdd(stats + 2, direct);
        atomicMax(stats + 3, deepest);
        atomicAdd(stats + 4, splits);
    }
}

}  // namespace

void hold_iota(int n, int* idx, cudaStream_t st) {
    if (n > 0) (k_hold_iota<<<grid_for(n, 256), 256, 0, st>>>(n, idx), note_launch());
}

void hold_gather(int k, const int* idx, const double* x, const double* y, const double* z, const double* vx,
                 const double* vy, const double* vz, const double* m, double* out, int stride, int zero_from,
                 cudaStream_t st) {
    if (k > 0)
        (k_hold_gather<<<grid_for(k, 256), 256, 0, st>>>(k, idx, x, y, z, vx, vy, vz, m, out, stride, zero_from),
         note_launch());
}

void hold_split(int k, const int* idx, const double* tau, double dt, uint32_t* flag, uint32_t* scan, int* S, int* F,
                uint32_t* nfast, uint32_t* scratch, cudaStream_t st) {
    if (k <= 0) return;
    (k_hold_flags<<<grid_for(k, 256), 256, 0, st>>>(k, tau, dt, flag), note_launch());
    cudaMemcpyAsync(scan, flag, 4 * (size_t)k, cudaMemcpyDeviceToDevice, st);
    scan_exclusive_u32_large(scan, k, nfast, scratch, st);
    (k_hold_compact<<<grid_for(k, 256), 256, 0, st>>>(k, idx, flag, scan, S, F), note_launch());
}

void hold_kick(int k, const int* idx, const double* acc, const double* sub, int stride, int sub_stride, double h,
               double* vx, double* vy, double* vz, cudaStream_t st) {
    if (k > 0)
        (k_hold_kick<<<grid_for(k, 256), 256, 0, st>>>(k, idx, acc, sub, stride, sub_stride, h, vx, vy, vz),
         note_launch());
}

void hold_drift(int k, const int* idx, double dt, double* x, double* y, double* z, const double* vx,
                const double* vy, const double* vz, cudaStream_t st) {
    if (k > 0) (k_hold_drift<<<grid_for(k, 256), 256, 0, st>>>(k, idx, dt, x, y, z, vx, vy, vz), note_launch());
}

size_t hold_small_smem(int k) {
    const size_t W = (size_t)(k + 31) / 32;
    return 10 * sizeof(double) * (size_t)k + hold_term_bytes(k) + sizeof(HoldFrame) * kHoldMaxLevels + 2 * sizeof(int) * (size_t)k +
           sizeof(unsigned) * W * kHoldMaxLevels;
}

void hold_small(int k, const int* idx, double* x, double* y, double* z, double* vx, double* vy, double* vz,
                const double* m, double G, double soft, double eta, bool sym, double dt, double dt_min, int depth,
                unsigned long long* stats, cudaStream_t st) {
    if (k <= 0) return;
    const size_t sh = hold_small_smem(k);
    auto go = [&](auto kernel, int most) {
        ensure_dyn_smem((const void*)kernel, (int)hold_small_smem(most));
        (kernel<<<1, kHoldThreads, sh, st>>>(k, idx, x, y, z, vx, vy, vz, m, G, soft * soft, eta, sym ? 1 : 0, dt,
                                             dt_min, depth, stats),
         note_launch());
    };
    if (k <= kHoldWhole) go(k_hold_small<false>, kHoldWhole);
    else go(k_hold_small<true>, kHoldSmallMax);
}

}  // namespace gbfmm
