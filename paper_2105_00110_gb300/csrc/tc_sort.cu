// Sort of the canonical edge keys by most significant digits: partition
// passes whose order within a bucket is free, then one local sort a bucket.
//
// A radix sort from the least significant digit moves every key once per
// digit (six passes for 48-bit keys), each pass stable, so a key's place in
// its tile takes a ranking over the warp.  From the most significant digit
// nothing has to be stable: a shared atomic gives a key a place among its
// tile's keys of the same digit and one global atomic a tile and digit
// reserves their place in the bucket.  Two passes bring 2^28 keys to buckets
// of about 512, which a CTA sorts in shared memory and writes back in place:
//
//   level   digit histogram (the first comes with the keys), offsets per
//           segment (k_seg_scan), scatter through a shared tile
//           (k_scatter) into the other buffer
//   bucket  at most kLocalCap keys: k_sort_tiny or k_sort_local; more (hub
//           rows): a segment of the next level, with the next digit
//
// Levels go on while such segments are left and bits remain; a segment whose
// bits are used up holds equal keys only.  Every bucket ends in the same
// buffer at its place, so the buffer is the sorted array.  Keys of all ones
// (self-loops) are dropped by the first scatter.
#include <algorithm>
#include <utility>

#include "tc_internal.cuh"

namespace tcx {

namespace {

typedef unsigned long long ull;
constexpr unsigned FULL = 0xffffffffu;

constexpr int kPartThreads = 512;
constexpr int kPartKeys = 16;                            // keys a thread holds
constexpr int kTile = kPartThreads * kPartKeys;          // 64 KB of keys
constexpr int kMaxDigit = 10;                            // bits of a digit: at least 8 keys a bin and tile
constexpr int kMaxBins = 1 << kMaxDigit;
constexpr int kLocalSmall = 1024;                        // keys of a 128-thread local sort
constexpr int kLocalCap = 4096;                          // ... of a 512-thread one
constexpr int kTargetBucket = 512;

// The segments of a level: segment k is keys [start[k], start[k] + size[k]),
// its tiles [tile[k], tile[k + 1]).
struct segments {
    const int64_t* start;
    const int64_t* size;
    const int64_t* tile;
    int64_t count;
};

__device__ __forceinline__ int64_t segment_of(const segments& sg, int64_t t, int lane) {
    int64_t lo = 0, hi = sg.count;   // last k with tile[k] <= t, 32 probes at a time
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) >> 5, x = lo + lane * step;
        const unsigned m = __ballot_sync(FULL, x < hi && sg.tile[x] <= t) | 1u;
        lo += (31 - __clz(m)) * step;
        hi = hi < lo + step ? hi : lo + step;
    }
    return lo;
}

// tile[k]: tiles before segment k, tile[count] all of them (one CTA)
__global__ void __launch_bounds__(1024) k_seg_tiles(const int64_t* __restrict__ size, int64_t count,
                                                    int64_t* __restrict__ tile) {
    __shared__ ull s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ull carry = 0;
    for (int64_t k0 = 0; k0 < count; k0 += 1024) {
        const int64_t k = k0 + threadIdx.x;
        const ull mine = k < count ? (ull)((size[k] + kTile - 1) / kTile) : 0;
        ull incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const ull y = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        ull before = 0, total = 0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const ull y = s_warp[j];
            before += j < warp ? y : 0;
            total += y;
        }
        if (k < count) tile[k] = (int64_t)(carry + before + incl - mine);
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) tile[count] = (int64_t)carry;
}

// Counts of digit (key >> shift) & (bins - 1) per segment.  A CTA takes a
// contiguous share of the tiles and adds its counts when the segment changes.
__global__ void __launch_bounds__(kPartThreads)
k_seg_hist(const uint64_t* __restrict__ keys, segments sg, int shift, int bins, uint32_t* __restrict__ cnt) {
    __shared__ uint32_t h[kMaxBins];
    __shared__ int64_t s_seg;
    for (int b = threadIdx.x; b < bins; b += kPartThreads) h[b] = 0;
    const int64_t tiles = sg.tile[sg.count];
    const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
    if (t0 >= t1) return;
    if (threadIdx.x < 32) {
        const int64_t k = segment_of(sg, t0, threadIdx.x);
        if (threadIdx.x == 0) s_seg = k;
    }
    __syncthreads();
    int64_t seg = s_seg;
    bool any = false;
    auto flush = [&] {
        __syncthreads();
        for (int b = threadIdx.x; b < bins; b += kPartThreads) {
            if (h[b]) atomicAdd(&cnt[seg * bins + b], h[b]);
            h[b] = 0;
        }
        __syncthreads();
    };
    for (int64_t t = t0; t < t1; ++t) {
        while (t >= sg.tile[seg + 1]) {
            if (any) flush();
            any = false;
            ++seg;
        }
        const int64_t off = (t - sg.tile[seg]) * kTile, left = sg.size[seg] - off;
        const uint64_t* src = keys + sg.start[seg] + off;
#pragma unroll
        for (int i = 0; i < kPartKeys; ++i) {
            const int j = i * kPartThreads + threadIdx.x;
            if (j < left) atomicAdd(&h[(src[j] >> shift) & (bins - 1)], 1u);
        }
        any = true;
    }
    if (any) flush();
}

// Counts of a segment -> its buckets: start and size of each, and the cursor
// the scatter reserves from.  One CTA a segment.
__global__ void __launch_bounds__(kMaxBins)
k_seg_scan(const uint32_t* __restrict__ cnt, segments sg, int bins, int64_t* __restrict__ start,
           int64_t* __restrict__ size, ull* __restrict__ cursor, int64_t* __restrict__ total) {
    __shared__ uint32_t s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t k = blockIdx.x; k < sg.count; k += gridDim.x) {
        const uint32_t mine = (int)threadIdx.x < bins ? cnt[k * bins + threadIdx.x] : 0;
        uint32_t incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        uint32_t before = 0, all = 0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const uint32_t y = s_warp[j];
            before += j < warp ? y : 0;
            all += y;
        }
        if ((int)threadIdx.x < bins) {
            const int64_t b = k * bins + threadIdx.x, at = sg.start[k] + before + incl - mine;
            start[b] = at;
            size[b] = mine;
            cursor[b] = (ull)at;
        }
        if (total && threadIdx.x == 0) *total = all;
        __syncthreads();
    }
}

// One tile at a time: a key's place among the tile's keys of its digit by a
// shared atomic, the bins' places in the tile by a scan, room for each bin in
// its bucket by one global atomic, then the tile is put together in shared
// memory and copied out bin by bin.  Bound by the copy (each key read and
// written once): 2^28 keys take 1.3 ms a pass, 3.4 TB/s; a stable pass of a
// least-significant-digit sort took 2.5.  FIRST: keys of all ones are dropped.
template <bool FIRST>
__global__ void __launch_bounds__(kPartThreads, 2)
k_scatter(const uint64_t* __restrict__ keys, uint64_t* __restrict__ out, segments sg, int shift, int bins,
          ull* __restrict__ cursor) {
    constexpr int T = kPartThreads, N = kPartKeys;
    extern __shared__ __align__(16) uint8_t part_dyn[];
    uint64_t* stage = (uint64_t*)part_dyn;               // [kTile]
    int64_t* base = (int64_t*)(stage + kTile);           // [kMaxBins] out position of the tile's key 0 of the bin
    uint32_t* h = (uint32_t*)(base + kMaxBins);          // [kMaxBins] keys per bin, then first key of it in the tile
    __shared__ uint32_t s_warp[T / 32];
    __shared__ int64_t s_seg;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tiles = sg.tile[sg.count];
    const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
    if (t0 >= t1) return;
    if (threadIdx.x < 32) {
        const int64_t k = segment_of(sg, t0, threadIdx.x);
        if (threadIdx.x == 0) s_seg = k;
    }
    __syncthreads();
    int64_t seg = s_seg;
    for (int64_t t = t0; t < t1; ++t) {
        while (t >= sg.tile[seg + 1]) ++seg;
        const int64_t off = (t - sg.tile[seg]) * kTile, left = sg.size[seg] - off, at = sg.start[seg] + off;
        uint64_t x[N];
        uint32_t place[N / 2];   // two 16-bit places each
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int j = i * T + threadIdx.x;
            x[i] = j < left ? keys[at + j] : ~0ull;
        }
        for (int b = threadIdx.x; b < bins; b += T) h[b] = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const bool in = FIRST ? x[i] != ~0ull : i * T + (int)threadIdx.x < left;
            const uint32_t p = in ? atomicAdd(&h[(x[i] >> shift) & (bins - 1)], 1u) : 0xffffu;
            if (i & 1) place[i >> 1] |= p << 16;
            else place[i >> 1] = p;
        }
        __syncthreads();
        // kMaxBins / T bins a thread
        constexpr int PB = kMaxBins / T;
        uint32_t c[PB], sum = 0;
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            const int b = PB * threadIdx.x + i;
            c[i] = b < bins ? h[b] : 0;
            sum += c[i];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += v;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        uint32_t run = incl - sum, n = 0;
#pragma unroll
        for (int j = 0; j < T / 32; ++j) {
            const uint32_t v = s_warp[j];
            run += j < warp ? v : 0;
            n += v;
        }
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            const int b = PB * threadIdx.x + i;
            if (b < bins) {
                h[b] = run;
                if (c[i]) base[b] = (int64_t)atomicAdd(&cursor[seg * bins + b], (ull)c[i]) - run;
            }
            run += c[i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint32_t p = (place[i >> 1] >> ((i & 1) * 16)) & 0xffffu;
            if (p != 0xffffu) stage[h[(x[i] >> shift) & (bins - 1)] + p] = x[i];
        }
        __syncthreads();
        for (uint32_t j = threadIdx.x; j < n; j += T) {
            const uint64_t k = stage[j];
            out[base[(k >> shift) & (bins - 1)] + j] = k;
        }
        __syncthreads();
    }
}

// Buckets by what sorts them: nothing (one key in place is sorted too, but
// is copied like the others), a warp, the small or the large local sort, or
// the next level.  Lists of bucket indices; counts in num[0..3].  `bits`: key
// bits below the digit (0: equal keys, which any list's kernel copies).
__global__ void k_bucket_lists(const int64_t* __restrict__ start, const int64_t* __restrict__ size, int64_t count,
                               int bits, int32_t* __restrict__ tiny, int32_t* __restrict__ small,
                               int32_t* __restrict__ large, int64_t* __restrict__ big_start,
                               int64_t* __restrict__ big_size, unsigned int* __restrict__ num) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t k0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 32; k0 < count; k0 += warps * 32) {
        const int64_t k = k0 + lane;
        const int64_t s = k < count ? size[k] : 0;
        const int c = s == 0 ? -1 : s <= 32 ? 0 : s <= kLocalSmall ? 1 : s <= kLocalCap || bits == 0 ? 2 : 3;
        for (int q = 0; q < 4; ++q) {
            const unsigned m = __ballot_sync(FULL, c == q);
            if (!m) continue;
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&num[q], (unsigned)__popc(m));
            at = __shfl_sync(FULL, at, 0) + __popc(m & ((1u << lane) - 1));
            if (c != q) continue;
            if (q == 0) tiny[at] = (int32_t)k;
            else if (q == 1) small[at] = (int32_t)k;
            else if (q == 2) large[at] = (int32_t)k;
            else {
                big_start[at] = start[k];
                big_size[at] = s;
            }
        }
    }
}

// A bucket of at most CAP keys, sorted by one CTA from `in` to the same
// place of `out` (they may be the same buffer).  Keys are grouped by their top bits below the bucket's (kGroups of them: rows of
// the lower end, mostly); a group of c keys gets c sub-bins, spread evenly
// between its smallest and its largest key, so that sub-bins hold about one
// key whether a group is one hub's row or a few light ones (float arithmetic
// is monotonic, so the order of sub-bins is the order of keys).  Keys go to
// their sub-bins, unordered within one, as in the scatter; a key's place
// there is the number of smaller keys, counted by reading it.  A bucket with
// a sub-bin of more than kCrowded keys takes a bitonic network instead.
// Bound by the latency of its steps, nine CTAs an SM: 2^28 R-MAT keys take
// 3.4 + 1.4 ms (both sizes), a fixed digit for the sub-bins, which left a hub
// row's keys in a few, 5.3 + 1.3.
constexpr uint32_t kCrowded = 128;
constexpr int kGroupBits = 8, kGroups = 1 << kGroupBits;
template <int T, int CAP>
__global__ void __launch_bounds__(T)
k_sort_local(const uint64_t* __restrict__ in, uint64_t* __restrict__ out, const int64_t* __restrict__ start,
             const int64_t* __restrict__ size, const int32_t* __restrict__ list, const unsigned int* __restrict__ num,
             int bits) {
    constexpr int N = CAP / T, PG = kGroups > T ? kGroups / T : 1;
    extern __shared__ __align__(16) uint8_t local_dyn[];
    uint64_t* key = (uint64_t*)local_dyn;        // [CAP]
    uint32_t* h = (uint32_t*)(key + CAP);        // [CAP + 4] keys per sub-bin, then the first of it
    __shared__ uint32_t g_cnt[kGroups], g_base[kGroups], g_min[kGroups], g_max[kGroups];
    __shared__ float g_scale[kGroups];
    __shared__ uint32_t s_warp[T / 32], s_most;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int gshift = bits > kGroupBits ? bits - kGroupBits : 0;
    const int rshift = gshift > 32 ? gshift - 32 : 0;   // the rest of a key in 32 bits
    const uint64_t rmask = ((uint64_t)1 << gshift) - 1;
    auto group = [&](uint64_t k) { return (uint32_t)(k >> gshift) & (kGroups - 1); };
    auto rest = [&](uint64_t k) { return (uint32_t)((k & rmask) >> rshift); };
    auto subbin = [&](uint64_t k) {
        const uint32_t g = group(k), c = g_cnt[g];
        const uint32_t i = (uint32_t)((float)(rest(k) - g_min[g]) * g_scale[g]);
        return g_base[g] + (i < c ? i : c - 1);
    };
    const unsigned count = *num;
    for (unsigned q = blockIdx.x; q < count; q += gridDim.x) {
        const int64_t k = list[q], s0 = start[k], s64 = size[k];
        if (bits == 0 || s64 == 1) {   // equal keys, any number of them
            if (in != out)
                for (int64_t j = t; j < s64; j += T) {
                    out[s0 + j] = in[s0 + j];
                }
            continue;
        }
        const int s = (int)s64;
        uint64_t x[N];
        uint32_t place[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            x[i] = i * T + t < s ? in[s0 + i * T + t] : 0;
        }
        for (int b = t; b < kGroups; b += T) {
            g_cnt[b] = 0;
            g_min[b] = 0xffffffffu;
            g_max[b] = 0;
        }
        for (int b = t; b < s; b += T) h[b] = 0;
        if (t == 0) s_most = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i * T + t < s) {
                const uint32_t g = group(x[i]), r = rest(x[i]);
                atomicAdd(&g_cnt[g], 1u);
                atomicMin(&g_min[g], r);
                atomicMax(&g_max[g], r);
            }
        __syncthreads();
        // places of the groups' sub-bins, PG groups a thread
        {
            uint32_t c[PG], sum = 0;
#pragma unroll
            for (int i = 0; i < PG; ++i) {
                const int g = t * PG + i;
                c[i] = g < kGroups ? g_cnt[g] : 0;
                sum += c[i];
            }
            uint32_t incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t v = __shfl_up_sync(FULL, incl, d);
                if (lane >= d) incl += v;
            }
            if (lane == 31) s_warp[warp] = incl;
            __syncthreads();
            uint32_t run = incl - sum;
            for (int j = 0; j < warp; ++j) run += s_warp[j];
#pragma unroll
            for (int i = 0; i < PG; ++i) {
                const int g = t * PG + i;
                if (g < kGroups) {
                    g_base[g] = run;
                    g_scale[g] = (float)c[i] / ((float)(g_max[g] - g_min[g]) + 1.0f);
                    run += c[i];
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i * T + t < s) {
                const uint32_t b = subbin(x[i]);
                place[i] = atomicAdd(&h[b], 1u) | (b << 16);   // both below CAP <= 4096
            }
        __syncthreads();
        {
            uint32_t c[N], sum = 0, most = 0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                c[i] = t * N + i < s ? h[t * N + i] : 0;
                sum += c[i];
                most = c[i] > most ? c[i] : most;
            }
            uint32_t incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t v = __shfl_up_sync(FULL, incl, d);
                if (lane >= d) incl += v;
            }
            most = __reduce_max_sync(FULL, most);
            if (lane == 31) s_warp[warp] = incl;
            if (lane == 0 && most > kCrowded) atomicMax(&s_most, most);
            __syncthreads();
            uint32_t run = incl - sum;
            for (int j = 0; j < warp; ++j) run += s_warp[j];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                if (t * N + i < s) h[t * N + i] = run;
                run += c[i];
            }
            if (t == 0) h[s] = (uint32_t)s;
        }
        __syncthreads();
        const bool crowded = s_most > kCrowded;
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i * T + t < s) {
                const uint32_t p = h[place[i] >> 16] + (place[i] & 0xffffu);
                key[p] = x[i];
            }
        __syncthreads();
        if (!crowded) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int j = i * T + t;
                if (j >= s) break;
                const uint64_t v = key[j];
                const uint32_t b = subbin(v);
                const int f = (int)h[b], e = (int)h[b + 1];
                int p = f;
                for (int r = f; r < e; ++r) {
                    const uint64_t z = key[r];
                    p += z < v || (z == v && r < j);
                }
                out[s0 + p] = v;
            }
        } else {
            int P = 1;
            while (P < s) P <<= 1;
            for (int m = 2; m <= P; m <<= 1)
                for (int d = m >> 1; d > 0; d >>= 1) {
                    const int ld = __ffs(d) - 1;
                    for (int u = t; u < (P >> 1); u += T) {
                        // the first step of a merge pairs mirror images, so the
                        // smaller key always goes to the lower index and a
                        // bucket sorts as if padded with +inf
                        const int a = ((u >> ld) << (ld + 1)) | (u & (d - 1));
                        const int b = d == (m >> 1) ? a ^ (m - 1) : a | d;
                        if (b < s) {
                            const uint64_t xa = key[a], xb = key[b];
                            if (xb < xa) {
                                key[a] = xb;
                                key[b] = xa;
                            }
                        }
                    }
                    __syncthreads();
                }
            for (int j = t; j < s; j += T) {
                out[s0 + j] = key[j];
            }
        }
        __syncthreads();
    }
}

// Buckets of at most 32 keys, a warp each (big segments leave millions of
// them): a key a lane, its place counted over the others.
__global__ void __launch_bounds__(256)
k_sort_tiny(const uint64_t* __restrict__ in, uint64_t* __restrict__ out, const int64_t* __restrict__ start,
            const int64_t* __restrict__ size, const int32_t* __restrict__ list, const unsigned int* __restrict__ num) {
    const int lane = threadIdx.x & 31;
    const unsigned count = *num, warps = gridDim.x * (blockDim.x >> 5);
    for (unsigned q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < count; q += warps) {
        const int32_t k = list[q];
        const int64_t s0 = start[k];
        const int s = (int)size[k];
        const uint64_t x = lane < s ? in[s0 + lane] : ~0ull;
        int p = 0;
        for (int r = 0; r < s; ++r) {
            const uint64_t z = __shfl_sync(FULL, x, r);
            p += z < x || (z == x && r < lane);
        }
        if (lane < s) out[s0 + p] = x;
    }
}

constexpr size_t part_smem() { return (size_t)kTile * 8 + kMaxBins * 12; }
constexpr size_t local_smem(int cap) { return (size_t)cap * 12 + 16; }

}  // namespace

// Digits of the first two levels together: buckets of about kTargetBucket.
static int digits_wanted(int64_t np) {
    int want = 0;
    while (want < 2 * kMaxDigit && ((int64_t)kTargetBucket << want) < np) ++want;
    return want;
}

int sort_first_digit(int64_t np, int bits) {
    const int want = digits_wanted(np);
    return std::min(bits, want <= kMaxDigit ? want : want / 2);
}

tc_status sort_keys_msd(const sort_alloc& get, uint64_t* keys, uint64_t* other, uint32_t* first_counts, int64_t np,
                        int bits, const unsigned int* err, uint64_t** sorted, int64_t* valid, cudaStream_t s) {
    // shared-memory limits (of the current device, so set on each call)
    TC_CUDA(cudaFuncSetAttribute(k_scatter<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)part_smem()));
    TC_CUDA(cudaFuncSetAttribute(k_scatter<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)part_smem()));
    TC_CUDA(cudaFuncSetAttribute(k_sort_local<512, kLocalCap>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)local_smem(kLocalCap)));
    const int want = digits_wanted(np), d0 = sort_first_digit(np, bits), sms = sm_count();
    int64_t *one = nullptr, *total = nullptr;
    unsigned int* num = nullptr;
    TC_TRY(get((void**)&one, 4 * 8));        // start, size and tiles of the whole array
    TC_TRY(get((void**)&total, 8));
    TC_TRY(get((void**)&num, 4 * 4));
    const int64_t h_one[4] = {0, np, 0, (np + kTile - 1) / kTile};
    TC_CUDA(cudaMemcpyAsync(one, h_one, sizeof(h_one), cudaMemcpyHostToDevice, s));
    segments sg{one, one + 1, one + 2, 1};
    uint64_t *src = keys, *dst = other;
    uint32_t* cnt = first_counts;
    int left = bits, digit = d0;
    *sorted = nullptr;
    for (int level = 0;; ++level) {
        const int64_t buckets = sg.count << digit;
        const int shift = left - digit, bins = 1 << digit;
        int64_t *bstart = nullptr, *bsize = nullptr;
        ull* cursor = nullptr;
        TC_TRY(get((void**)&bstart, buckets * 8));
        TC_TRY(get((void**)&bsize, buckets * 8));
        TC_TRY(get((void**)&cursor, buckets * 8));
        if (level > 0) {
            TC_TRY(get((void**)&cnt, buckets * 4));
            TC_CUDA(cudaMemsetAsync(cnt, 0, buckets * 4, s));
            launch_scope ls("build_sort_hist", s);
            k_seg_hist<<<sms * 4, kPartThreads, 0, s>>>(src, sg, shift, bins, cnt);
            TC_LAUNCH_CHECK();
        }
        {
            launch_scope ls("build_sort_scan", s);
            k_seg_scan<<<(int)std::min<int64_t>(sg.count, sms * 8), kMaxBins, 0, s>>>(
                cnt, sg, bins, bstart, bsize, cursor, level == 0 ? total : nullptr);
            TC_LAUNCH_CHECK();
        }
        {
            launch_scope ls("build_sort_scatter", s);
            if (level == 0)
                k_scatter<true><<<sms * 2, kPartThreads, part_smem(), s>>>(src, dst, sg, shift, bins, cursor);
            else
                k_scatter<false><<<sms * 2, kPartThreads, part_smem(), s>>>(src, dst, sg, shift, bins, cursor);
            TC_LAUNCH_CHECK();
        }
        left = shift;
        std::swap(src, dst);
        if (level == 0 && want > d0 && left > 0) {   // every bucket goes on
            int64_t* tiles = nullptr;
            TC_TRY(get((void**)&tiles, (buckets + 1) * 8));
            launch_scope ls("build_sort_tiles", s);
            k_seg_tiles<<<1, 1024, 0, s>>>(bsize, buckets, tiles);
            TC_LAUNCH_CHECK();
            sg = segments{bstart, bsize, tiles, buckets};
            digit = std::min(left, std::min(want - d0, kMaxDigit));
            continue;
        }
        int32_t *tiny = nullptr, *small = nullptr, *large = nullptr;
        int64_t *big_start = nullptr, *big_size = nullptr;
        const int64_t most_big = np / kLocalCap + 1;
        TC_TRY(get((void**)&tiny, buckets * 4));
        TC_TRY(get((void**)&small, buckets * 4));
        TC_TRY(get((void**)&large, buckets * 4));
        TC_TRY(get((void**)&big_start, most_big * 8));
        TC_TRY(get((void**)&big_size, most_big * 8));
        TC_CUDA(cudaMemsetAsync(num, 0, 4 * 4, s));
        {
            launch_scope ls("build_sort_lists", s);
            const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((buckets + 255) / 256, sms * 8));
            k_bucket_lists<<<blocks, 256, 0, s>>>(bstart, bsize, buckets, left, tiny, small, large, big_start,
                                                  big_size, num);
            TC_LAUNCH_CHECK();
        }
        if (!*sorted) *sorted = src;   // the first buckets' buffer holds the result
        {
            launch_scope ls("build_sort_tiny", s);
            k_sort_tiny<<<sms * 8, 256, 0, s>>>(src, *sorted, bstart, bsize, tiny, num);
            TC_LAUNCH_CHECK();
        }
        {
            launch_scope ls("build_sort_small", s);
            k_sort_local<128, kLocalSmall><<<sms * 12, 128, local_smem(kLocalSmall), s>>>(src, *sorted, bstart, bsize,
                                                                                          small, num + 1, left);
            TC_LAUNCH_CHECK();
        }
        {
            launch_scope ls("build_sort_large", s);
            k_sort_local<512, kLocalCap><<<sms * 3, 512, local_smem(kLocalCap), s>>>(src, *sorted, bstart, bsize,
                                                                                    large, num + 2, left);
            TC_LAUNCH_CHECK();
        }
        unsigned int h_num[4] = {0, 0, 0, 0}, h_err = 0;
        int64_t h_total = 0;
        TC_CUDA(cudaMemcpyAsync(h_num, num, 16, cudaMemcpyDeviceToHost, s));
        TC_CUDA(cudaMemcpyAsync(&h_total, total, 8, cudaMemcpyDeviceToHost, s));
        TC_CUDA(cudaMemcpyAsync(&h_err, err, 4, cudaMemcpyDeviceToHost, s));
        TC_CUDA(cudaStreamSynchronize(s));
        if (h_err) return TC_ERR_INVALID_ARG;
        *valid = h_total;
        const int64_t bigs = (int64_t)h_num[3];
        if (bigs == 0) return TC_OK;
        int64_t* tiles = nullptr;
        TC_TRY(get((void**)&tiles, (bigs + 1) * 8));
        launch_scope ls("build_sort_tiles", s);
        k_seg_tiles<<<1, 1024, 0, s>>>(big_size, bigs, tiles);
        TC_LAUNCH_CHECK();
        sg = segments{big_start, big_size, tiles, bigs};
        digit = std::min(left, kMaxDigit);
    }
}

}  // namespace tcx
