// Stable LSD radix sort of 64- or 32-bit keys with optional 32-bit payloads.
//
// One kernel counts the digits of every pass, then one kernel per 8-bit digit
// moves the keys. A block takes tiles by ticket, ranks each key among the
// earlier keys of its tile with the same digit (warp match + per-warp digit
// counters), so equal keys keep their order, and learns where the tile's digits
// go from a decoupled look-back over the earlier tiles' published counts: one
// thread per digit, four records at a time. Every key is read and written once
// per pass. (Decoupled look-back: Merrill and Garland, "Single-pass parallel prefix
// scan with decoupled look-back", 2016; one sweep per digit: Adinets and Merrill,
// "Onesweep: a faster least significant digit radix sort for GPUs", 2022.)
//
// What bounds it: ranking and the scattered writes where there are many tiles;
// the launch where there are few. With a histogram, its scan (one or three
// launches) and a scatter per pass, the 8 passes over 4096 body keys took 200 us
// of kernels, then 91, now 43 (k_sort_tile); all sorts of 2^20 bodies (8 passes of bodies, 12 of list
// keys) 1.67 ms, now 1.20.
//
// Waits are bounded (about a second): a block that gives up raises kErrTimeout
// in the sort's error word and goes on with the prefix it has; its positions
// stay inside the array, and the users of the sorted data check the word or
// clamp what they read (the host then fails the call). Once the word is raised,
// later waits last a millisecond.
#include "gbfmm_internal.cuh"

namespace gbfmm {

namespace {
constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 8;                    // keys per thread
constexpr int kTile = kThreads * kItems;     // 4096 keys per block
constexpr int kWarpItems = kTile / kWarps;   // 256 contiguous keys per warp
constexpr int kMaxPasses = 8;
template <typename K, bool VAL>
constexpr size_t scatter_smem() {
    return (size_t)kTile * (sizeof(K) + (VAL ? 4 : 0)) + (size_t)(kWarps + 2) * 256 * 4;
}
// Blocks per SM the pass kernel's registers are cut for (40, a few spills for
// 64-bit keys): a pass is a chain of waits (loads, ranks, look-back), so warps
// in flight count. With 16 keys per thread of 256 and two blocks, 16 warps on an SM,
// the 16 passes over the 64-bit list keys of 8M bodies took 8.4 ms, now 5.1 (16 keys a
// thread in blocks of 512: faster there, .21 ms slower on its 8 passes over the bodies).
constexpr int kPassBlocks = 3;

// Scratch of a sort: digit counts of every pass, a tile ticket per pass (both
// zeroed before the sort), then the look-back records, 256 per tile: bits 63-62
// the kind (1: the tile's own count, 2: its inclusive prefix), 61-56 the pass, the
// rest the value, so one load reads a consistent record. The count kernel clears
// the records; the pass field tells a pass's records from the last one's.
constexpr size_t kSortHeadWords = 256 * kMaxPasses + kMaxPasses;
struct SortScratch {
    uint32_t* digits;   // [pass][256]
    uint32_t* tickets;  // [pass]
    unsigned long long* rec;
    __host__ __device__ explicit SortScratch(uint32_t* w)
        : digits(w), tickets(w + 256 * kMaxPasses), rec(reinterpret_cast<unsigned long long*>(w + kSortHeadWords)) {}
};
static_assert(kSortHeadWords % 2 == 0, "the records are 8-byte aligned");

constexpr unsigned long long kRecCount = 1ull << 62, kRecPrefix = 2ull << 62;
constexpr unsigned long long kRecValue = (1ull << 56) - 1ull;
constexpr unsigned long long kSortWaitNs = 1000000000ull;      // one second
constexpr unsigned long long kSortWaitFailedNs = 1000000ull;   // when a wait before has run out

__device__ __forceinline__ void rec_store(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long rec_load(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned err_load(const unsigned* p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long sort_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Digit counts of all passes in one read of the keys (the counts do not depend
// on the order), and clear look-back records.
template <typename K>
__global__ void __launch_bounds__(kThreads) k_sort_count(const K* __restrict__ keys, int64_t n,
                                                         const unsigned long long* __restrict__ dn, int lo_bit,
                                                         int npass, SortScratch s) {
    __shared__ uint32_t h[kMaxPasses * 256];
    if (dn && (int64_t)*dn < n) n = (int64_t)*dn;
    const int64_t ntiles = (n + kTile - 1) / kTile;
    for (int i = threadIdx.x; i < npass * 256; i += kThreads) h[i] = 0;
    __syncthreads();
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        if (threadIdx.x < 256) s.rec[t * 256 + threadIdx.x] = 0ull;
        K key[kItems];
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const int64_t i = t * kTile + (int64_t)k * kThreads + threadIdx.x;
            key[k] = i < n ? keys[i] : K(0);
        }
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const bool valid = t * kTile + (int64_t)k * kThreads + threadIdx.x < n;
            const unsigned act = __ballot_sync(0xffffffffu, valid);
            for (int p = 0; p < npass; ++p) {
                const unsigned d = (unsigned)(key[k] >> (lo_bit + 8 * p)) & 255u;
                // a warp of one digit (the leading digits of neighbouring keys) counts it at once
                const unsigned d0 = __shfl_sync(0xffffffffu, d, 0);
                if (__all_sync(0xffffffffu, !valid || d == d0)) {
                    if ((threadIdx.x & 31) == 0 && act) atomicAdd(&h[p * 256 + d0], (uint32_t)__popc(act));
                } else if (valid) {
                    atomicAdd(&h[p * 256 + d], 1u);
                }
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < npass * 256; i += kThreads)
        if (h[i]) atomicAdd(s.digits + i, h[i]);
}

// inclusive scan of v over the warp
__device__ __forceinline__ uint32_t warp_scan(uint32_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Rank of each of the thread's keys among the warp's earlier keys with the same
// digit (two 16-bit ranks to a word); count (zero before): the warp's keys per digit.
template <typename K>
__device__ __forceinline__ void rank_items(const K* key, int mine, int shift, uint32_t* count, int lane,
                                           uint32_t* rank) {
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const bool valid = 32 * r < mine;
        const uint32_t d = valid ? (uint32_t)(key[r] >> shift) & 255u : 0xFFFFFFFFu;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = valid ? count[d] : 0u;
        const uint32_t rk = before + __popc(peers & ((1u << lane) - 1u));
        rank[r / 2] = r % 2 ? rank[r / 2] | rk << 16 : rk;
        __syncwarp();
        if (valid && lane == 31 - __clz(peers)) count[d] = before + __popc(peers);
        __syncwarp();
    }
}

template <typename K, bool VAL>
__global__ void __launch_bounds__(kThreads, kPassBlocks) k_sort_pass(
    const K* __restrict__ kin, const uint32_t* __restrict__ vin, K* __restrict__ kout, uint32_t* __restrict__ vout,
    int64_t n, const unsigned long long* __restrict__ dn, int shift, int pass, SortScratch s, unsigned* err,
    int stall) {
    extern __shared__ __align__(16) unsigned char sh_scatter[];
    K* skey = reinterpret_cast<K*>(sh_scatter);                                  // kTile
    uint32_t* sval = reinterpret_cast<uint32_t*>(skey + kTile);                  // kTile (VAL only)
    uint32_t (*wcount)[256] = reinterpret_cast<uint32_t (*)[256]>(sval + (VAL ? kTile : 0));  // kWarps x 256
    uint32_t* boff = &wcount[kWarps][0];    // global start of each digit for this tile
    uint32_t* lstart = boff + 256;          // start of each digit inside the tile
    __shared__ unsigned s_tile;
    __shared__ uint32_t s_wsum[2][kWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) s_tile = atomicAdd(s.tickets + pass, 1u);
    for (int i = threadIdx.x; i < kWarps * 256; i += kThreads) (&wcount[0][0])[i] = 0;
    __syncthreads();
    const int64_t tile = s_tile;
    const int64_t tile0 = tile * kTile;
    if (dn && (int64_t)*dn < n) n = (int64_t)*dn;
    if (tile0 >= n) return;  // the whole block: nothing of this tile is present
    const int present = (int)(n - tile0 < kTile ? n - tile0 : kTile);
    const int mine = present - warp * kWarpItems - lane;  // item r of this thread is present if 32 r < mine
    kin += tile0 + warp * kWarpItems + lane;
    if (VAL) vin += tile0 + warp * kWarpItems + lane;
    K key[kItems];
    uint32_t val[VAL ? kItems : 1], rank[kItems / 2];  // (two 16-bit ranks to a word)
    // all loads first, so that they are in flight together
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        key[r] = 32 * r < mine ? kin[32 * r] : K(0);
        if (VAL) val[VAL ? r : 0] = 32 * r < mine ? vin[32 * r] : 0u;
    }
    const uint32_t digits_all = threadIdx.x < 256 ? s.digits[pass * 256 + threadIdx.x] : 0u;
    rank_items(key, mine, shift, wcount[warp], lane, rank);
    __syncthreads();
    // thread d < 256: the tile's count of digit d, published at once
    const int d = threadIdx.x;
    unsigned long long* rec = s.rec + d;
    const unsigned long long tag = (unsigned long long)pass << 56;
    uint32_t cnt = 0, gbase = 0;
    if (d < 256) {
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t t = wcount[w][d];
            wcount[w][d] = cnt;
            cnt += t;
        }
        rec_store(rec + tile * 256, (tile == 0 ? kRecPrefix : kRecCount) | tag | cnt);
    }
    // exclusive scans over the digits: the tile's counts and all keys' counts
    const uint32_t in_tile = warp_scan(cnt, lane), in_all = warp_scan(digits_all, lane);
    if (lane == 31) {
        s_wsum[0][warp] = in_tile;
        s_wsum[1][warp] = in_all;
    }
    __syncthreads();
    if (d < 256) {
        uint32_t lbase = in_tile - cnt;
        gbase = in_all - digits_all;
        for (int w = 0; w < warp; ++w) {
            lbase += s_wsum[0][w];
            gbase += s_wsum[1][w];
        }
        lstart[d] = lbase;
    }
    __syncthreads();
    // reorder the tile by digit in shared memory
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        if (32 * r < mine) {
            const uint32_t dd = (uint32_t)(key[r] >> shift) & 255u;
            const uint32_t pos = lstart[dd] + wcount[warp][dd] + (rank[r / 2] >> 16 * (r % 2) & 0xffffu);
            skey[pos] = key[r];
            if (VAL) sval[pos] = val[VAL ? r : 0];
        }
    }
    // look-back for digit d: the keys of it in the tiles before this one
    uint32_t excl = 0;
    if (tile > 0 && d < 256) {
        constexpr int kAhead = 4;
        const unsigned long long want = (tag >> 56) + (stall ? kMaxPasses : 0);  // (stall: of no record)
        unsigned long long t0 = 0;
        bool done = false;
        for (int64_t j = tile - 1; !done; j -= kAhead) {
            unsigned long long w[kAhead];
#pragma unroll
            for (int q = 0; q < kAhead; ++q) w[q] = j - q >= 0 ? rec_load(rec + (j - q) * 256) : (kRecPrefix | tag);
#pragma unroll
            for (int q = 0; q < kAhead; ++q) {
                if (!done) {
                    while ((w[q] >> 62) == 0ull || ((w[q] >> 56) & 63ull) != want) {
                        const unsigned long long now = sort_ns();
                        if (t0 == 0) t0 = now;
                        if (now - t0 > kSortWaitNs ||
                            (now - t0 > kSortWaitFailedNs && (err_load(err) & kErrTimeout))) {
                            atomicOr(err, kErrTimeout);
                            w[q] = kRecPrefix | tag;  // go on with what there is
                            break;
                        }
                        w[q] = rec_load(rec + (j - q) * 256);
                    }
                    excl += (uint32_t)(w[q] & kRecValue);
                    done = (w[q] >> 62) == 2ull;
                }
            }
        }
        rec_store(rec + tile * 256, kRecPrefix | tag | (excl + cnt));
    }
    if (d < 256) boff[d] = gbase + excl;
    __syncthreads();
    for (int j = threadIdx.x; j < present; j += kThreads) {
        const K k = skey[j];
        const uint32_t dd = (uint32_t)(k >> shift) & 255u;
        const uint32_t pos = boff[dd] + (uint32_t)j - lstart[dd];
        if ((int64_t)pos >= n) continue;  // (never: only a wait that ran out could misplace a key)
        kout[pos] = k;
        if (VAL) vout[pos] = sval[j];
    }
}

// All passes of one tile in one block, for up to kTile keys, in place: a pass is
// some 5 us of ranking and exchange in shared memory, where a launch of k_sort_pass
// takes 10. 4096 body keys with the permutation: 91 -> 43 us.
template <typename K, bool VAL>
__global__ void __launch_bounds__(kThreads) k_sort_tile(K* __restrict__ keys, uint32_t* __restrict__ vals, int64_t n,
                                                        const unsigned long long* __restrict__ dn, int lo_bit,
                                                        int npass) {
    extern __shared__ __align__(16) unsigned char sh_scatter[];
    K* skey = reinterpret_cast<K*>(sh_scatter);
    uint32_t* sval = reinterpret_cast<uint32_t*>(skey + kTile);
    uint32_t (*wcount)[256] = reinterpret_cast<uint32_t (*)[256]>(sval + (VAL ? kTile : 0));
    uint32_t* lstart = &wcount[kWarps][0];
    __shared__ uint32_t s_wsum[kWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, d = threadIdx.x;
    if (dn && (int64_t)*dn < n) n = (int64_t)*dn;
    const int first = warp * kWarpItems + lane;
    const int mine = (int)n - first;  // item r of this thread is present if 32 r < mine
    K key[kItems];
    uint32_t val[VAL ? kItems : 1], rank[kItems / 2];
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        key[r] = 32 * r < mine ? keys[first + 32 * r] : K(0);
        if (VAL) val[VAL ? r : 0] = 32 * r < mine ? vals[first + 32 * r] : 0u;
    }
    for (int pass = 0; pass < npass; ++pass) {
        const int shift = lo_bit + 8 * pass;
        for (int i = threadIdx.x; i < kWarps * 256; i += kThreads) (&wcount[0][0])[i] = 0;
        __syncthreads();
        rank_items(key, mine, shift, wcount[warp], lane, rank);
        __syncthreads();
        uint32_t cnt = 0;
        if (d < 256) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t t = wcount[w][d];
                wcount[w][d] = cnt;
                cnt += t;
            }
        }
        const uint32_t in_tile = warp_scan(cnt, lane);
        if (lane == 31) s_wsum[warp] = in_tile;
        __syncthreads();
        if (d < 256) {
            uint32_t lbase = in_tile - cnt;
            for (int w = 0; w < warp; ++w) lbase += s_wsum[w];
            lstart[d] = lbase;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kItems; ++r) {
            if (32 * r < mine) {
                const uint32_t dd = (uint32_t)(key[r] >> shift) & 255u;
                const uint32_t pos = lstart[dd] + wcount[warp][dd] + (rank[r / 2] >> 16 * (r % 2) & 0xffffu);
                skey[pos] = key[r];
                if (VAL) sval[pos] = val[VAL ? r : 0];
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kItems; ++r) {
            if (32 * r < mine) {
                key[r] = skey[first + 32 * r];
                if (VAL) val[VAL ? r : 0] = sval[first + 32 * r];
            }
        }
    }
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        if (32 * r < mine) {
            keys[first + 32 * r] = key[r];
            if (VAL) vals[first + 32 * r] = val[VAL ? r : 0];
        }
    }
}

// Single-block exclusive scan in tiles of 4096 words: a coalesced load into
// shared memory, four consecutive words per thread, a block scan of the
// thread sums, a coalesced store, and a carry into the next tile.
__global__ void __launch_bounds__(1024) k_scan(uint32_t* data, int64_t count, uint32_t* total) {
    __shared__ __align__(16) uint32_t tile[4096];
    __shared__ uint32_t warp_sums[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t carry = 0;
    for (int64_t base = 0; base < count; base += 4096) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = base + k * 1024 + tid;
            tile[k * 1024 + tid] = i < count ? data[i] : 0u;
        }
        __syncthreads();
        const uint4 v = reinterpret_cast<const uint4*>(tile)[tid];
        const uint32_t s = v.x + v.y + v.z + v.w;
        uint32_t incl = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const uint32_t ws = warp_sums[lane];
            uint32_t wi = ws;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += t;
            }
            warp_sums[lane] = wi - ws;  // exclusive offsets of the warps; the tile total is wi at lane 31
            if (lane == 31) tile[0] = wi;  // tile[0] was consumed above; reused to pass the total
        }
        __syncthreads();
        const uint32_t tile_total = tile[0];
        uint32_t run = carry + warp_sums[warp] + incl - s;
        __syncthreads();
        uint4 o;
        o.x = run; run += v.x;
        o.y = run; run += v.y;
        o.z = run; run += v.z;
        o.w = run;
        reinterpret_cast<uint4*>(tile)[tid] = o;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = base + k * 1024 + tid;
            if (i < count) data[i] = tile[k * 1024 + tid];
        }
        carry += tile_total;
        __syncthreads();
    }
    if (tid == 0 && total) *total = carry;
}
// Large scans in three passes: segment sums, a scan of the sums, and a
// rescan of each segment from its offset.
constexpr int kSegment = 4096;
__global__ void __launch_bounds__(256) k_seg_sum(const uint32_t* __restrict__ data, int64_t count,
                                                 uint32_t* __restrict__ sums) {
    __shared__ uint32_t red[256];
    const int64_t base = (int64_t)blockIdx.x * kSegment;
    uint32_t s = 0;
    for (int k = threadIdx.x; k < kSegment; k += 256) {
        const int64_t i = base + k;
        if (i < count) s += data[i];
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = red[0];
}

__global__ void __launch_bounds__(256) k_seg_scan(uint32_t* __restrict__ data, int64_t count,
                                                  const uint32_t* __restrict__ offs) {
    __shared__ uint32_t warp_sums[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * kSegment + (int64_t)threadIdx.x * (kSegment / 256);
    uint32_t v[kSegment / 256];
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < kSegment / 256; ++k) {
        const int64_t i = base + k;
        v[k] = i < count ? data[i] : 0u;
        s += v[k];
    }
    uint32_t incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    uint32_t wo = 0;
    for (int w = 0; w < warp; ++w) wo += warp_sums[w];
    uint32_t run = offs[blockIdx.x] + wo + incl - s;
#pragma unroll
    for (int k = 0; k < kSegment / 256; ++k) {
        const int64_t i = base + k;
        if (i < count) data[i] = run;
        run += v[k];
    }
}
}  // namespace

size_t scan_scratch_words(int64_t count) { return (size_t)((count + kSegment - 1) / kSegment + 2); }

void scan_exclusive_u32_large(uint32_t* data, int64_t count, uint32_t* total, uint32_t* scratch,
                              cudaStream_t st) {
    // one block scans 4096 values at a time, one tile after another: beyond a
    // few tiles the three parallel passes finish sooner
    if (count <= 4 * 4096) {
        (k_scan<<<1, 1024, 0, st>>>(data, count, total), note_launch());
        return;
    }
    const int nseg = (int)((count + kSegment - 1) / kSegment);
    (k_seg_sum<<<nseg, 256, 0, st>>>(data, count, scratch), note_launch());
    (k_scan<<<1, 1024, 0, st>>>(scratch, nseg, total), note_launch());
    (k_seg_scan<<<nseg, 256, 0, st>>>(data, count, scratch), note_launch());
}

size_t radix_hist_words(int64_t n) {
    const int64_t nb = (n + kTile - 1) / kTile;
    return kSortHeadWords + 2 * 256 * (size_t)(nb > 0 ? nb : 1);
}

void scan_exclusive_u32(uint32_t* data, int64_t count, uint32_t* total, cudaStream_t st) {
    (k_scan<<<1, 1024, 0, st>>>(data, count, total), note_launch());
}

namespace {
template <typename K, bool VAL>
int radix_sort_impl(K* k0, uint32_t* v0, K* k1, uint32_t* v1, int64_t n, int lo_bit, int bits, uint32_t* hist,
                    cudaStream_t st, const unsigned long long* dn, unsigned* err, bool stall) {
    if (n <= 1 || bits <= lo_bit) return 0;
    const int npass = (bits - lo_bit + 7) / 8;
    if (n <= kTile) {
        ensure_dyn_smem((const void*)k_sort_tile<K, VAL>, (int)scatter_smem<K, VAL>());
        (k_sort_tile<K, VAL><<<1, kThreads, scatter_smem<K, VAL>(), st>>>(k0, v0, n, dn, lo_bit, npass), note_launch());
        return 0;
    }
    ensure_dyn_smem((const void*)k_sort_pass<K, VAL>, (int)scatter_smem<K, VAL>());
    const int nblocks = (int)((n + kTile - 1) / kTile);
    const SortScratch s(hist);
    cudaMemsetAsync(hist, 0, sizeof(uint32_t) * kSortHeadWords, st);
    const int count_grid = nblocks < 4 * device_sm_count() ? nblocks : 4 * device_sm_count();
    (k_sort_count<K><<<count_grid, kThreads, 0, st>>>(k0, n, dn, lo_bit, npass, s), note_launch());
    int cur = 0;
    for (int pass = 0; pass < npass; ++pass) {
        K* ki = cur ? k1 : k0;
        uint32_t* vi = cur ? v1 : v0;
        K* ko = cur ? k0 : k1;
        uint32_t* vo = cur ? v0 : v1;
        (k_sort_pass<K, VAL><<<nblocks, kThreads, scatter_smem<K, VAL>(), st>>>(ki, vi, ko, vo, n, dn,
                                                                                lo_bit + 8 * pass, pass, s, err, stall ? 1 : 0),
         note_launch());
        cur ^= 1;
    }
    return cur;
}
}  // namespace

int radix_sort(uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, int64_t n, int bits, uint32_t* hist,
               unsigned* err, cudaStream_t st, const unsigned long long* dn, int lo_bit, bool stall) {
    return v0 ? radix_sort_impl<uint64_t, true>(k0, v0, k1, v1, n, lo_bit, bits, hist, st, dn, err, stall)
              : radix_sort_impl<uint64_t, false>(k0, nullptr, k1, nullptr, n, lo_bit, bits, hist, st, dn, err, stall);
}

int radix_sort32(uint32_t* k0, uint32_t* k1, int64_t n, int bits, uint32_t* hist, unsigned* err, cudaStream_t st,
                 const unsigned long long* dn, int lo_bit, bool stall) {
    return radix_sort_impl<uint32_t, false>(k0, nullptr, k1, nullptr, n, lo_bit, bits, hist, st, dn, err, stall);
}

}  // namespace gbfmm
