// tc_build_csr: simple undirected graph, degree order π, orientation and
// the count-step plan, all on the device.
//
//  1. pairs -> canonical keys (min, max); self-loops become a sentinel
//     (the set-up of section "Comparison": symmetrised, loop-free, simple)
//  2. sort (tc_sort.cu; small inputs: CUB) + unique -> the m undirected
//     edges, caller labels
//  3. degrees; π = sort by (degree, label) (section "Notation")
//  4. every edge relabelled by π and placed in the run of its lower end;
//     each run sorted (warp registers, a warp's shared region or a CTA,
//     by length) -> symmetric CSR in rank space whose rows are
//     [N_L(v) | N_H(v)] (Lemma 1's partition), N_H(v) ascending
//  5. written with the runs: col, edge_tail, and the head record
//     {u, hrem, twin} of every lower neighbour
//  6. planner: per middle vertex v its work W(v) = Σ_{u∈N_L(v)} hrem, and
//     the work items of the count step, heavy vertices split into chunks
//
// The radix sorts of small inputs and of the degree order, the unique step
// and the scans use CUB (header-only, compiled into this library); the per-row
// run sorts are this file's own.
#include <cub/cub.cuh>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "tc_internal.cuh"

namespace tcx {

namespace {

constexpr int kThreads = 256;
constexpr int64_t kMsdPairs = 1 << 19;            // pairs from which the keys are sorted by tc_sort.cu
constexpr int64_t kMaxDegreeReadBack = 1 << 20;   // vertices above which the largest degree is read back

inline int grid_for(int64_t n, int per_thread = 1) {
    int64_t want = (n + (int64_t)kThreads * per_thread - 1) / ((int64_t)kThreads * per_thread);
    int64_t cap = (int64_t)sm_count() * 16;
    if (want < 1) want = 1;
    return (int)std::min(want, cap);
}

// One chunk of `chunk` items a block, however many blocks: blocks start in
// order, so the items in work at a time are neighbours and what they scatter
// to nearby places meets in L2.  (A grid of 16 CTAs an SM striding over all
// items sweeps them two to three times, each sweep touching every place: the
// 8192-graph batch's edges took 12.4 ms to scatter that way, 7.3 in order.)
inline int ordered_blocks(int64_t n, int64_t chunk) { return (int)std::max<int64_t>(1, (n + chunk - 1) / chunk); }

#define GRID_STRIDE(i, n) \
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

// Pairs -> canonical keys (lower label, higher label), ~0 for a self-loop or
// a bad id.  With cnt, also how many keys have each value of their top
// bits (key >> shift, `bins` of them): the first digit of the sort.
struct digit_counts {
    uint32_t* cnt;   // null: not wanted
    int shift, bins;
};
constexpr int kMaxFirstBins = 1024;
__device__ __forceinline__ void digit_add(const digit_counts& dc, uint32_t* h, uint64_t key) {
    if (dc.cnt && key != ~0ull) atomicAdd(&h[key >> dc.shift], 1u);
}
__device__ __forceinline__ void digit_begin(const digit_counts& dc, uint32_t* h) {
    if (!dc.cnt) return;
    for (int b = threadIdx.x; b < dc.bins; b += blockDim.x) h[b] = 0;
    __syncthreads();
}
__device__ __forceinline__ void digit_end(const digit_counts& dc, uint32_t* h) {
    if (!dc.cnt) return;
    __syncthreads();
    for (int b = threadIdx.x; b < dc.bins; b += blockDim.x)
        if (h[b]) atomicAdd(&dc.cnt[b], h[b]);
}

template <typename T>
__global__ void k_make_keys(const T* __restrict__ src, const T* __restrict__ dst, int64_t np,
                            int64_t n, int bits, uint64_t* __restrict__ keys,
                            unsigned int* __restrict__ err, digit_counts dc) {
    __shared__ uint32_t h[kMaxFirstBins];
    digit_begin(dc, h);
    GRID_STRIDE(i, np) {
        int64_t a = (int64_t)src[i], b = (int64_t)dst[i];
        uint64_t key = ~0ull;
        if (a < 0 || b < 0 || a >= n || b >= n) {
            atomicOr(err, 1u);
        } else if (a != b) {
            uint64_t lo = (uint64_t)(a < b ? a : b), hi = (uint64_t)(a < b ? b : a);
            key = (lo << bits) | hi;
        }
        keys[i] = key;
        digit_add(dc, h, key);
    }
    digit_end(dc, h);
}

// The same for a union's pairs (ids local to their graph): a warp takes
// kUnionChunk consecutive pairs, finds the graph of the first and steps on
// from there.  An edge lies inside one graph, so the key holds the lower
// label and the distance of the higher one in dbits bits (the same order in
// fewer bits).  (A search per pair into shifted copies, keyed in a second
// launch, took 3.2 ms on the 8192-graph batch.)
constexpr int kUnionChunk = 32 * 32;
template <typename T>
__global__ void k_make_union_keys(const T* __restrict__ src, const T* __restrict__ dst, int64_t np, union_layout un,
                                  int dbits, uint64_t* __restrict__ keys, unsigned int* __restrict__ err,
                                  digit_counts dc) {
    __shared__ uint32_t h[kMaxFirstBins];
    digit_begin(dc, h);
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t chunks = (np + kUnionChunk - 1) / kUnionChunk;
    bool bad = false;
    for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c < chunks; c += warps) {
        const int64_t i0 = c * kUnionChunk, i1 = i0 + kUnionChunk < np ? i0 + kUnionChunk : np;
        int64_t k = 0, hi = un.G;   // last k with poff[k] <= i0, 32 probes at a time
        while (hi - k > 1) {
            const int64_t step = (hi - k + 31) >> 5, x = k + lane * step;
            const unsigned m = __ballot_sync(0xffffffffu, x < hi && un.poff[x] <= i0) | 1u;
            k += (31 - __clz(m)) * step;
            hi = hi < k + step ? hi : k + step;
        }
        int64_t p1 = un.poff[k + 1], v0 = un.voff[k], nk = un.voff[k + 1] - v0;
        for (int64_t i = i0 + lane; i < i1; i += 32) {
            while (i >= p1) {   // i < np = poff[G]: ends at a graph with pairs
                ++k;
                p1 = un.poff[k + 1];
                v0 = un.voff[k];
                nk = un.voff[k + 1] - v0;
            }
            const int64_t a = (int64_t)src[i], b = (int64_t)dst[i];
            uint64_t key = ~0ull;
            if (a < 0 || b < 0 || a >= nk || b >= nk) bad = true;
            else if (a < b) key = ((uint64_t)(v0 + a) << dbits) | (uint64_t)(b - a);
            else if (b < a) key = ((uint64_t)(v0 + b) << dbits) | (uint64_t)(a - b);
            keys[i] = key;
            digit_add(dc, h, key);
        }
    }
    digit_end(dc, h);
    if (bad) atomicOr(err, 1u);
}

// sel[0] unique keys, the last of them all ones if there were loops -> the
// edges, and the error word in sel[1]: one copy and one wait for what were
// three and two (R-MAT scale 12 569 -> 542 us a pass).
__global__ void k_edge_count(const uint64_t* __restrict__ uniq, const unsigned int* __restrict__ err,
                             int64_t* __restrict__ sel) {
    const int64_t k = sel[0];
    sel[0] = k > 0 && uniq[k - 1] == ~0ull ? k - 1 : k;
    sel[1] = *err;
}

// Canonical keys -> edge list and degrees; the low `bits` hold the higher
// end, or (delta) its distance from the lower one.
__global__ void k_edges_degrees(const uint64_t* __restrict__ ukeys, int64_t m, int bits, bool delta,
                                int32_t* __restrict__ eu, int32_t* __restrict__ ev,
                                int32_t* __restrict__ deg) {
    const uint64_t mask = (1ull << bits) - 1;
    GRID_STRIDE(e, m) {
        uint64_t k = ukeys[e];
        int32_t u = (int32_t)(k >> bits), v = (int32_t)(k & mask) + (delta ? u : 0);
        eu[e] = u;
        ev[e] = v;
        // edges are sorted by u: lanes with the same u add their count once
        const unsigned same = __match_any_sync(__activemask(), u);
        if ((threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&deg[u], __popc(same));
        atomicAdd(&deg[v], 1);
    }
}

__global__ void k_max_degree(const int32_t* __restrict__ deg, int64_t n, int32_t* __restrict__ out) {
    int32_t x = 0;
    GRID_STRIDE(v, n) x = max(x, deg[v]);
    x = __reduce_max_sync(0xffffffffu, x);
    if ((threadIdx.x & 31) == 0 && x) atomicMax(out, x);
}

// Graph of every label of a union, a warp per 32·kLabelRounds labels.
constexpr int kLabelRounds = 32;
__global__ void k_label_graph(union_layout un, int64_t n, int32_t* __restrict__ lg) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5), per = 32 * kLabelRounds;
    for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c * per < n; c += warps) {
        const int64_t v0 = c * per, v1 = v0 + per < n ? v0 + per : n;
        int64_t k = 0, hi = un.G;
        while (hi - k > 1) {
            const int64_t step = (hi - k + 31) >> 5, x = k + lane * step;
            const unsigned m = __ballot_sync(0xffffffffu, x < hi && un.voff[x] <= v0) | 1u;
            k += (31 - __clz(m)) * step;
            hi = hi < k + step ? hi : k + step;
        }
        for (int64_t v = v0 + lane; v < v1; v += 32) {
            while (v >= un.voff[k + 1]) ++k;
            lg[v] = (int32_t)k;
        }
    }
}

// Sort keys of the degree order π (section "Notation"): the degree; the
// sort is stable and the labels come in order, so ties go by label.  A union
// sorts by (graph, degree): within a graph that is the degree order, and the
// only edges are within a graph, so every result is the same, while a graph's
// vertices have neighbouring ranks: what the build scatters and the count and
// gather read at random stays in L2, and the id windows of N_H(v) are those
// of the graph alone.
struct rank_key {
    int dbits;   // bits of a degree
    int gshift;  // graphs of a union taken 2^gshift at a time (all bits fit 32)
    int gbits;   // bits of the shifted graph index (0: no union)
};
__global__ void k_rank_keys(const int32_t* __restrict__ deg, int64_t n, rank_key rk, const int32_t* __restrict__ lg,
                            uint32_t* __restrict__ keys, int32_t* __restrict__ labels, int64_t* __restrict__ band) {
    if (blockIdx.x == 0 && threadIdx.x < 2) band[threadIdx.x] = lg ? 0 : n;   // set by k_rank_apply
    GRID_STRIDE(v, n) {
        const int32_t d = deg[v];
        uint32_t k = (uint32_t)d;
        if (rk.gbits) k |= ((uint32_t)lg[v] >> rk.gshift) << rk.dbits;
        keys[v] = k;
        labels[v] = (int32_t)v;
    }
}

// Rows of degree up to 32, up to TC_BAND_CTA (mid) and above (hubs) take a
// thread, a warp and a CTA each in the gather, and likewise in the per-row
// work.  Where degrees ascend with rank, band[k] is the first rank above
// limit k (n if none): the rank whose degree is the first to pass it.  A
// union (lg) lists its mid rows from list[0] and its hubs from list[hub_at],
// counted in band; the order of a list is of no account.
#ifndef TC_BAND_CTA
#define TC_BAND_CTA 4096
#endif
__device__ __forceinline__ int degree_band(int32_t d) { return d <= 32 ? 0 : d <= TC_BAND_CTA ? 1 : 2; }
__global__ void k_rank_apply(const uint32_t* __restrict__ sorted, const int32_t* __restrict__ labels, int64_t n,
                             int dbits, const int32_t* __restrict__ lg, int32_t* __restrict__ perm,
                             int32_t* __restrict__ rank, int64_t* __restrict__ degr, int32_t* __restrict__ rank_graph,
                             int64_t* __restrict__ band, int32_t* __restrict__ list, int64_t hub_at) {
    const uint32_t mask = dbits < 32 ? (1u << dbits) - 1 : 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // whole warps step together (the lists' places are taken warp by warp)
    GRID_STRIDE(r, (n + 31) & ~31ll) {
        int32_t d = 0;
        if (r < n) {
            const int32_t v = labels[r];
            perm[r] = v;
            rank[v] = (int32_t)r;
            d = (int32_t)(sorted[r] & mask);
            degr[r] = d;
            if (lg) rank_graph[r] = lg[v];
        }
        if (!lg) {
            if (d > 32) {
                const int32_t before = r ? (int32_t)(sorted[r - 1] & mask) : 0;
                if (before <= 32) band[0] = r;
                if (d > TC_BAND_CTA && before <= TC_BAND_CTA) band[1] = r;
            }
            continue;
        }
        for (int k = 0; k < 2; ++k) {
            const bool in = d > 32 && (d > TC_BAND_CTA) == (k == 1);
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (!m) continue;
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd((unsigned long long*)&band[k], (unsigned long long)__popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (in) list[(k ? hub_at : 0) + (int64_t)at + __popc(m & ((1u << lane) - 1))] = (int32_t)r;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) degr[n] = 0;
}

// Every undirected edge once in rank space: key (lo, hi) with lo < hi the
// ranks of its ends, at its canonical id; d_H(lo) counted.
__global__ void k_edge_rank_keys(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                                 const int32_t* __restrict__ rank, int64_t m, int bits,
                                 uint64_t* __restrict__ keys, int32_t* __restrict__ dh) {
    GRID_STRIDE(e, m) {
        const uint64_t ru = (uint64_t)rank[eu[e]], rv = (uint64_t)rank[ev[e]];
        const uint64_t lo = ru < rv ? ru : rv, hi = ru < rv ? rv : ru;
        keys[e] = (lo << bits) | hi;
        atomicAdd(&dh[lo], 1);
    }
}

// Row split: the last d_H(r) entries of row r hold N_H(r).  The head cursor
// of row r starts at its first entry (an absolute CSR position), its
// tail-run cursor at hptr[r] (the run's start in the compact tail order).
template <class C>
__global__ void k_hstart(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ dh,
                         const int64_t* __restrict__ hptr, int64_t n, int64_t* __restrict__ hstart,
                         C* __restrict__ hnext, C* __restrict__ tnext, int64_t* __restrict__ work) {
    GRID_STRIDE(r, n) {
        work[r] = 0;   // k_row_work adds to it
        hstart[r] = row_ptr[r + 1] - dh[r];
        hnext[r] = (C)row_ptr[r];
        tnext[r] = (C)hptr[r];
    }
}

// Each edge to the next free slot of its lower end's run (row r's run
// starts at hptr[r]) as (hi << 32) | edge id, so that sorting each run puts
// N_H(lo) in order with the edge ids alongside.  A block takes
// kThreads * kPlace consecutive edges, kPlace cursor atomics a thread in flight.
constexpr int kPlace = 4;
template <class C>
__global__ void __launch_bounds__(kThreads)
k_tail_place(const uint64_t* __restrict__ keys, int64_t m, int bits, C* __restrict__ tnext,
             uint64_t* __restrict__ slot) {
    const uint64_t mask = (1ull << bits) - 1;
    const int64_t e0 = blockIdx.x * (int64_t)(kThreads * kPlace) + threadIdx.x;
    uint64_t k[kPlace];
    int64_t at[kPlace];
#pragma unroll
    for (int j = 0; j < kPlace; ++j)
        if (e0 + j * kThreads < m) k[j] = keys[e0 + j * kThreads];
#pragma unroll
    for (int j = 0; j < kPlace; ++j)
        if (e0 + j * kThreads < m) at[j] = (int64_t)atomicAdd(&tnext[k[j] >> bits], (C)1);
#pragma unroll
    for (int j = 0; j < kPlace; ++j)
        if (e0 + j * kThreads < m) slot[at[j]] = ((k[j] & mask) << 32) | (uint64_t)(e0 + j * kThreads);
}

// Both entries of one edge, from the i-th element x of row r's sorted run
// (tail position t = hstart[r] + i): the tail entry col[t] = hi, the edge's
// canonical id -> t, and the head entry in row hi (N_L(hi) in any order) at
// the next free slot of its cursor, as the record
// {r, |{w ∈ N_H(r) : w > hi}| = e - t - 1, twin = t}.
template <class C>
__device__ __forceinline__ void write_tail(int64_t r, int64_t t, int64_t e, uint64_t x, int64_t hp,
                                           int32_t* __restrict__ col, tc_head* __restrict__ head,
                                           C* __restrict__ edge_tail, int64_t core_t) {
    col[t] = (int32_t)(x >> 32);
    edge_tail[x & 0xffffffffull] = (C)t;
    tc_head rec;
    rec.u = (int32_t)r;
    // a lower end in the dense core (ranks >= core_t) streams nothing: the
    // core's product counts those triangles
    rec.hrem = r >= core_t ? 0 : (int32_t)(e - t - 1);
    rec.twin = t;
    store_head(head + hp, rec);
}

template <class C>
__device__ __forceinline__ void emit_tail(int64_t r, int64_t t, int64_t e, uint64_t x, C* __restrict__ hnext,
                                          int32_t* __restrict__ col, tc_head* __restrict__ head,
                                          C* __restrict__ edge_tail, int64_t core_t) {
    const int64_t hp = (int64_t)atomicAdd(&hnext[(int32_t)(x >> 32)], (C)1);
    write_tail(r, t, e, x, hp, col, head, edge_tail, core_t);
}

// Every run is sorted by bitonic merges in the form whose compare-exchanges
// all put the smaller key at the lower index: the first step of the k-merge
// pairs i with its mirror in the k-block (i ^ (k - 1)), the later steps pair
// i with i ^ j.  A run of length L sorts as if padded with +inf up to a
// power of two, since every pair whose upper index is >= L is a no-op; no
// padding is stored.
__device__ __forceinline__ uint64_t shfl_xor64(uint64_t x, int m) {
    const uint32_t lo = __shfl_xor_sync(0xffffffffu, (uint32_t)x, m);
    const uint32_t hi = __shfl_xor_sync(0xffffffffu, (uint32_t)(x >> 32), m);
    return ((uint64_t)hi << 32) | lo;
}

// One step (merge k, distance j) of the network over key[0, len), padded to
// P, by the threads t0, t0 + nt, ... of a team.
__device__ __forceinline__ void run_network_step(uint64_t* key, int len, int P, int k, int j, int t0, int nt) {
    const int lj = __ffs(j) - 1;
    for (int t = t0; t < (P >> 1); t += nt) {
        const int a = ((t >> lj) << (lj + 1)) | (t & (j - 1));
        const int b = j == (k >> 1) ? a ^ (k - 1) : a | j;
        if (b < len) {
            const uint64_t xa = key[a], xb = key[b];
            if (xb < xa) {
                key[a] = xb;
                key[b] = xa;
            }
        }
    }
}

// Runs of 33..kMidShort tails are sorted by one warp, kMidShort+1..kMidRun
// by one CTA of kMidWarps warps, longer ones by a CTA in shared memory (or
// in place); the first two in registers (below), with the shared-memory
// networks of k_runs_mid kept as the alternative.
constexpr int kMidRun = 1024;
#ifndef TC_MID_SHORT
#define TC_MID_SHORT 256
#endif
constexpr int kMidShort = TC_MID_SHORT;   // longest run of the one-warp tier (512 spilled: slower)

// Runs of 1..32 tails.  A warp takes 32 rows at a time and walks their runs as
// one concatenation, a tail a lane: the higher ends go to shared memory, and
// a tail's place in its run is the number of smaller ones there (they are
// distinct), counted by reading the run, whose lanes share those reads.  So
// every lane works however short the runs are, and four tails' cursor atomics
// and stores a lane are in flight together.  Bound by those scattered stores,
// a sector each in L2 and DRAM (more of them in flight a lane changed nothing);
// a network over the warp's registers, eight
// runs at a time with a run in the first lanes of each register, kept 3 of 32
// lanes busy on the 8192-graph batch (4096^2 grid: 6.4 -> 5.6 ms; with the
// blocks in order 4.5, and 12.3 -> 7.1 on the batch; with head records stored
// whole 4.4 and 6.5).
// Longer runs are queued: 33..kMidShort tails from the front of `big`
// (count nbig[0]) and kMidShort+1..kMidRun tails from the back of its first
// n entries (count nbig[1]) for k_runs_mid, which never meet since there are
// at most n runs; more than kMidRun tails after those n entries for
// k_runs_big (count nbig[2], fewer than m / kMidRun).
constexpr int kSmallTails = 512;   // tails a warp holds at a time
// A warp takes 32 rows from this many rows an SM on, where they fill the
// device's warps, and four below, in CTAs of one warp: the 4096 rows of R-MAT
// scale 12 were 128 warps on 16 SMs (36 -> 12 us; scale 16, 431 rows an SM, 44 -> 38).
constexpr int64_t kSmallRowsFrom = 1024;
struct small_runs {
    int64_t p0[32];      // first tail of each row's run in slot
    int64_t hs[32];      // row split: first tail position
    int64_t re[32];      // row end
    int32_t pre[32];     // tails before each row in this round
    int32_t hi[kSmallTails];
    uint8_t row[kSmallTails];
};
template <class C>
__global__ void __launch_bounds__(kThreads)
k_runs_small(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ hstart,
             const int64_t* __restrict__ hptr, const uint64_t* __restrict__ slot, int64_t n,
             C* __restrict__ hnext, int32_t* __restrict__ col, tc_head* __restrict__ head,
             C* __restrict__ edge_tail, int32_t* __restrict__ big,
             unsigned int* __restrict__ nbig, int64_t core_t, int rows) {
    __shared__ small_runs s_runs[kThreads / 32];
    small_runs& sr = s_runs[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t base = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * rows; base < n;
         base += warps * rows) {
        const int64_t r = base + lane;
        int len = 0;
        if (lane < rows && r < n) {
            const int64_t p0 = hptr[r], L = hptr[r + 1] - p0;
            if (L > kMidRun) big[n + (int64_t)atomicAdd(&nbig[2], 1u)] = (int32_t)r;
            else if (L > kMidShort) big[n - 1 - (int64_t)atomicAdd(&nbig[1], 1u)] = (int32_t)r;
            else if (L > 32) big[atomicAdd(&nbig[0], 1u)] = (int32_t)r;
            else if (L > 0) {
                len = (int)L;
                sr.p0[lane] = p0;
                sr.hs[lane] = hstart[r];
                sr.re[lane] = row_ptr[r + 1];
            }
        }
        int incl = len;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += x;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        // rounds of whole rows with at most kSmallTails tails (at least 16 rows)
        for (int done = 0; done < total;) {
            const int end = (int)__reduce_max_sync(0xffffffffu, incl <= done + kSmallTails ? (unsigned)incl : 0u);
            const int T = end - done;
            sr.pre[lane] = incl - len - done;   // negative for rows of earlier rounds
            __syncwarp();
            int at = 0;
            for (int j = lane; j < T; j += 32) {
                while (at < 31 && sr.pre[at + 1] <= j) ++at;
                sr.row[j] = (uint8_t)at;
                sr.hi[j] = (int32_t)(slot[sr.p0[at] + j - sr.pre[at]] >> 32);
            }
            __syncwarp();
            constexpr int K = 4;
            for (int j0 = lane; j0 < T; j0 += 32 * K) {
                uint64_t x[K];
                int64_t hp[K];
                int row[K], place[K];
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int j = j0 + 32 * k;
                    if (j < T) {
                        row[k] = sr.row[j];
                        const int f = sr.pre[row[k]];
                        x[k] = slot[sr.p0[row[k]] + j - f];
                        hp[k] = (int64_t)atomicAdd(&hnext[(int32_t)(x[k] >> 32)], (C)1);
                        const int32_t mine = (int32_t)(x[k] >> 32);
                        const int L = (int)(sr.re[row[k]] - sr.hs[row[k]]);
                        int c = 0;
                        for (int q = 0; q < L; ++q) c += sr.hi[f + q] < mine;
                        place[k] = c;
                    }
                }
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (j0 + 32 * k < T)
                        write_tail(base + row[k], sr.hs[row[k]] + place[k], sr.re[row[k]], x[k], hp[k], col, head,
                                   edge_tail, core_t);
            }
            __syncwarp();
            done = end;
        }
        __syncwarp();
    }
}

// Queued runs of 33..kMidShort tails (CAP = kMidShort: nbig[0] of them at
// the front of `big`) or kMidShort+1..kMidRun tails (CAP = kMidRun: nbig[1]
// at the back of its first n entries): one warp per run, the network in the
// warp's own shared region of CAP keys.
constexpr int kMidWarps = 4;

template <class C, int CAP>
__global__ void __launch_bounds__(32 * kMidWarps)
k_runs_mid(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ hstart,
           const int64_t* __restrict__ hptr, const uint64_t* __restrict__ slot, const int32_t* __restrict__ big,
           const unsigned int* __restrict__ nbig, int64_t n, C* __restrict__ hnext, int32_t* __restrict__ col,
           tc_head* __restrict__ head, C* __restrict__ edge_tail, int64_t core_t) {
    static_assert(CAP == kMidShort || CAP == kMidRun, "one queue per capacity");
    static_assert(kMidShort == 256 || kMidShort == 512, "register sort tiers: up to 16 keys a lane");
    constexpr bool kBack = CAP == kMidRun;
    __shared__ uint64_t sk[kMidWarps][CAP];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint64_t* key = sk[w];
    const unsigned count = nbig[kBack ? 1 : 0];
    const unsigned warps = gridDim.x * kMidWarps;
    for (unsigned q = blockIdx.x * kMidWarps + w; q < count; q += warps) {
        const int64_t r = kBack ? big[n - 1 - (int64_t)q] : big[q];
        const int64_t i0 = hptr[r];
        const int len = (int)(hptr[r + 1] - i0);
        for (int i = lane; i < len; i += 32) key[i] = slot[i0 + i];
        __syncwarp();
        int P = 1;
        while (P < len) P <<= 1;
        for (int k = 2; k <= P; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                run_network_step(key, len, P, k, j, lane, 32);
                __syncwarp();
            }
        const int64_t h = hstart[r], e = row_ptr[r + 1];
        for (int i = lane; i < len; i += 32) emit_tail(r, h + i, e, key[i], hnext, col, head, edge_tail, core_t);
        __syncwarp();
    }
}

// Runs of 33..kMidShort tails sorted in registers instead (TC_RUNS_REG):
// key i of the run (i = 32 e + lane, e < E) in register e of a lane, padded
// with +inf to 32 E.  Compare-exchanges at distance j < 32 pair lanes
// (shuffles), at j >= 32 pair registers of one lane; the mirror step of a
// k-merge pairs i with i ^ (k - 1), i.e. lane ^ (k - 1) for k <= 32 and
// register e ^ ((k - 1) >> 5) of lane ^ 31 above.  Loads and the emit's
// col stores are coalesced (lane-consecutive), and no shared memory is used.
#ifndef TC_RUNS_REG
#define TC_RUNS_REG 1
#endif
template <int E>
__device__ __forceinline__ void sort_run_regs(uint64_t (&x)[E], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1) {
        if (k <= 32) {
            const bool low = (lane & (k >> 1)) == 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint64_t y = shfl_xor64(x[e], k - 1);
                x[e] = low ? (x[e] < y ? x[e] : y) : (x[e] < y ? y : x[e]);
            }
        } else {
            // registers e (lower half of the k-block) and f = e ^ m pair with
            // each other's values in lane ^ 31
            const int m = (k - 1) >> 5;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int f = e ^ m;
                if (e < f) {
                    const uint64_t a = shfl_xor64(x[f], 31), b = shfl_xor64(x[e], 31);
                    x[e] = x[e] < a ? x[e] : a;   // e has bit k/64 clear: the lower index
                    x[f] = x[f] < b ? b : x[f];
                }
            }
        }
#pragma unroll
        for (int j = k >> 2; j > 0; j >>= 1) {
            if (j < 32) {
                const bool low = (lane & j) == 0;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint64_t y = shfl_xor64(x[e], j);
                    x[e] = low ? (x[e] < y ? x[e] : y) : (x[e] < y ? y : x[e]);
                }
            } else {
                const int je = j >> 5;
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if ((e & je) == 0) {
                        const uint64_t a = x[e], b = x[e | je];
                        x[e] = a < b ? a : b;
                        x[e | je] = a < b ? b : a;
                    }
            }
        }
    }
}

template <class C, int E>
__device__ __forceinline__ void run_regs(int lane, int64_t r, int64_t i0, int len, const uint64_t* __restrict__ slot,
                                         int64_t h, int64_t end, C* __restrict__ hnext, int32_t* __restrict__ col,
                                         tc_head* __restrict__ head, C* __restrict__ edge_tail, int64_t core_t) {
    uint64_t x[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = 32 * e + lane;
        x[e] = i < len ? slot[i0 + i] : ~0ull;
    }
    sort_run_regs<E>(x, lane);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = 32 * e + lane;
        if (i < len) emit_tail(r, h + i, end, x[e], hnext, col, head, edge_tail, core_t);
    }
}

template <class C>
__global__ void __launch_bounds__(32 * kMidWarps)
k_runs_mid_reg(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ hstart,
               const int64_t* __restrict__ hptr, const uint64_t* __restrict__ slot, const int32_t* __restrict__ big,
               const unsigned int* __restrict__ nbig, C* __restrict__ hnext, int32_t* __restrict__ col,
               tc_head* __restrict__ head, C* __restrict__ edge_tail, int64_t core_t) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned count = nbig[0];
    const unsigned warps = gridDim.x * kMidWarps;
    for (unsigned q = blockIdx.x * kMidWarps + w; q < count; q += warps) {
        const int64_t r = big[q];
        const int64_t i0 = hptr[r];
        const int len = (int)(hptr[r + 1] - i0);
        const int64_t h = hstart[r], end = row_ptr[r + 1];
        if (len <= 64) run_regs<C, 2>(lane, r, i0, len, slot, h, end, hnext, col, head, edge_tail, core_t);
        else if (len <= 128) run_regs<C, 4>(lane, r, i0, len, slot, h, end, hnext, col, head, edge_tail, core_t);
        else if (kMidShort <= 256 || len <= 256) run_regs<C, 8>(lane, r, i0, len, slot, h, end, hnext, col, head, edge_tail, core_t);
        else run_regs<C, (kMidShort > 256 ? 16 : 8)>(lane, r, i0, len, slot, h, end, hnext, col, head, edge_tail, core_t);
    }
}

// Runs of kMidShort+1..kMidRun tails by one CTA of kMidWarps warps in
// registers (TC_RUNS_CTA_REG): key i = 32 E w + 32 e + lane in register e of
// lane `lane` of warp w, padded with +inf to 128 E.  Distances below 32 pair
// lanes (shuffles), 32..32E-1 registers of one lane, 32E and above warps,
// through one shared exchange of all keys per such step.
#ifndef TC_RUNS_CTA_REG
#define TC_RUNS_CTA_REG 1
#endif
template <int E>
__device__ __forceinline__ void sort_run_cta(uint64_t (&x)[E], uint64_t* sx, int lane, int w) {
    constexpr int P = 32 * E * kMidWarps;
    const int me = 32 * E * w + lane;   // index of register 0
#pragma unroll
    for (int k = 2; k <= P; k <<= 1) {
        if (k <= 32) {
            const bool low = (lane & (k >> 1)) == 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint64_t y = shfl_xor64(x[e], k - 1);
                x[e] = low ? (x[e] < y ? x[e] : y) : (x[e] < y ? y : x[e]);
            }
        } else if (k <= 32 * E) {
            const int m = (k - 1) >> 5;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int f = e ^ m;
                if (e < f) {
                    const uint64_t a = shfl_xor64(x[f], 31), b = shfl_xor64(x[e], 31);
                    x[e] = x[e] < a ? x[e] : a;
                    x[f] = x[f] < b ? b : x[f];
                }
            }
        } else {
            // partner of i is i ^ (k - 1): another warp, register E-1-e, lane ^ 31
#pragma unroll
            for (int e = 0; e < E; ++e) sx[me + 32 * e] = x[e];
            __syncthreads();
            const int pw = w ^ ((k - 1) / (32 * E));
            const bool low = (w & (k / (64 * E))) == 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint64_t y = sx[32 * E * pw + 32 * (E - 1 - e) + (lane ^ 31)];
                x[e] = low ? (x[e] < y ? x[e] : y) : (x[e] < y ? y : x[e]);
            }
            __syncthreads();
        }
#pragma unroll
        for (int j = k >> 2; j > 0; j >>= 1) {
            if (j < 32) {
                const bool low = (lane & j) == 0;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint64_t y = shfl_xor64(x[e], j);
                    x[e] = low ? (x[e] < y ? x[e] : y) : (x[e] < y ? y : x[e]);
                }
            } else if (j < 32 * E) {
                const int je = j >> 5;
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if ((e & je) == 0) {
                        const uint64_t a = x[e], b = x[e | je];
                        x[e] = a < b ? a : b;
                        x[e | je] = a < b ? b : a;
                    }
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) sx[me + 32 * e] = x[e];
                __syncthreads();
                const int pw = w ^ (j / (32 * E));
                const bool low = (w & (j / (32 * E))) == 0;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint64_t y = sx[32 * E * pw + 32 * e + lane];
                    x[e] = low ? (x[e] < y ? x[e] : y) : (x[e] < y ? y : x[e]);
                }
                __syncthreads();
            }
        }
    }
}

template <class C, int E>
__device__ __forceinline__ void run_cta(int lane, int w, uint64_t* sx, int64_t r, int64_t i0, int len,
                                        const uint64_t* __restrict__ slot, int64_t h, int64_t end,
                                        C* __restrict__ hnext, int32_t* __restrict__ col,
                                        tc_head* __restrict__ head, C* __restrict__ edge_tail, int64_t core_t) {
    uint64_t x[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = 32 * E * w + 32 * e + lane;
        x[e] = i < len ? slot[i0 + i] : ~0ull;
    }
    sort_run_cta<E>(x, sx, lane, w);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = 32 * E * w + 32 * e + lane;
        if (i < len) emit_tail(r, h + i, end, x[e], hnext, col, head, edge_tail, core_t);
    }
}

template <class C>
__global__ void __launch_bounds__(32 * kMidWarps)
k_runs_long_cta(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ hstart,
                const int64_t* __restrict__ hptr, const uint64_t* __restrict__ slot, const int32_t* __restrict__ big,
                const unsigned int* __restrict__ nbig, int64_t n, C* __restrict__ hnext, int32_t* __restrict__ col,
                tc_head* __restrict__ head, C* __restrict__ edge_tail, int64_t core_t) {
    static_assert(32 * 8 * kMidWarps == kMidRun, "eight keys a thread cover the longest queued run");
    __shared__ uint64_t sx[kMidRun];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned count = nbig[1];
    for (unsigned q = blockIdx.x; q < count; q += gridDim.x) {
        const int64_t r = big[n - 1 - (int64_t)q];
        const int64_t i0 = hptr[r];
        const int len = (int)(hptr[r + 1] - i0);
        const int64_t h = hstart[r], end = row_ptr[r + 1];
        if (len <= 512) run_cta<C, 4>(lane, w, sx, r, i0, len, slot, h, end, hnext, col, head, edge_tail, core_t);
        else run_cta<C, 8>(lane, w, sx, r, i0, len, slot, h, end, hnext, col, head, edge_tail, core_t);
    }
}

// Queued runs longer than kMidRun (nbig[2] of them, after the first n
// entries of `big`): one CTA per run, the network in shared memory (up to
// kRunSmem keys) or in place in `slot`.
constexpr int kRunSmem = 4096;
constexpr int kRunThreads = 512;

template <class C>
__global__ void __launch_bounds__(kRunThreads)
k_runs_big(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ hstart,
           const int64_t* __restrict__ hptr, uint64_t* __restrict__ slot, const int32_t* __restrict__ big,
           const unsigned int* __restrict__ nbig, int64_t n, C* __restrict__ hnext, int32_t* __restrict__ col,
           tc_head* __restrict__ head, C* __restrict__ edge_tail, int64_t core_t) {
    __shared__ uint64_t sk[kRunSmem];
    const unsigned count = nbig[2];
    for (unsigned q = blockIdx.x; q < count; q += gridDim.x) {
        const int64_t r = big[n + (int64_t)q];
        const int64_t i0 = hptr[r];
        const int len = (int)(hptr[r + 1] - i0);
        uint64_t* key = len <= kRunSmem ? sk : slot + i0;
        if (len <= kRunSmem)
            for (int i = threadIdx.x; i < len; i += blockDim.x) sk[i] = slot[i0 + i];
        __syncthreads();
        int P = 1;
        while (P < len) P <<= 1;
        for (int k = 2; k <= P; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                run_network_step(key, len, P, k, j, threadIdx.x, blockDim.x);
                __syncthreads();
            }
        const int64_t h = hstart[r], e = row_ptr[r + 1];
        for (int i = threadIdx.x; i < len; i += blockDim.x) emit_tail(r, h + i, e, key[i], hnext, col, head, edge_tail, core_t);
        __syncthreads();
    }
}

// ------------------------------------------------------------ row work
struct row_stats {
    unsigned long long sum_h2, wedges, sum_dh, max_h, max_d;
};

// W(v) = Σ_{u ∈ N_L(v)} hrem(u, v), the number of ids the count step
// streams for middle vertex v, plus shape statistics.  One launch takes the
// mid rows with a warp each, the rows of degree up to 32 with a thread, and
// first the CSR positions of the hub rows (up to hundreds of thousands of
// head entries) in segments of kRowSegment, a warp each, added into work
// (zeroed beforehand): with a CTA a row the largest hub alone took 0.55 ms on
// the 4096^2 grid.  A union's hubs are few and apart: a CTA each.  It reads
// every head record once.  The statistics are reduced per CTA before the five atomics: with
// one set a warp, 10^5 atomics on five addresses took 33 + 18 us of the R-MAT
// scale-12 pass and 0.13 ms at scales 16 and 20.
constexpr int kRowWarps = kThreads / 32;
constexpr int64_t kRowSegment = 2048;
struct row_acc {
    unsigned long long h2 = 0, w = 0, dh = 0, maxh = 0, maxd = 0;
    __device__ __forceinline__ void add(unsigned long long hv, unsigned long long d, unsigned long long wr) {
        h2 += hv * hv;
        w += wr;
        dh += d * hv;
        maxh = maxh > hv ? maxh : hv;
        maxd = maxd > d ? maxd : d;
    }
    __device__ __forceinline__ void join(const row_acc& o) {
        h2 += o.h2;
        w += o.w;
        dh += o.dh;
        maxh = maxh > o.maxh ? maxh : o.maxh;
        maxd = maxd > o.maxd ? maxd : o.maxd;
    }
};

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long w) {
    for (int o = 16; o; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    return w;
}

__global__ void __launch_bounds__(kThreads)
k_row_work(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ hstart, const tc_head* __restrict__ head,
           const int64_t* __restrict__ band, const int32_t* __restrict__ list, int64_t hub_at, int64_t n,
           int64_t* __restrict__ work, row_stats* __restrict__ st) {
    __shared__ row_acc s_acc[kRowWarps];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int64_t b0 = band[0], b1 = band[1];
    const int64_t mids = list ? b0 : b1 - b0, smalls = list ? n : b0;
    const int64_t warps = (int64_t)gridDim.x * kRowWarps, w0 = (int64_t)blockIdx.x * kRowWarps + wp;
    row_acc acc;
    if (list) {
        for (int64_t k = blockIdx.x; k < b1; k += gridDim.x) {
            const int64_t r = list[hub_at + k], b = row_ptr[r], h = hstart[r], e = row_ptr[r + 1];
            unsigned long long w = 0;
#pragma unroll 4
            for (int64_t p = b + threadIdx.x; p < h; p += kThreads) w += (unsigned long long)head[p].hrem;
            w = warp_sum64(w);
            if (lane == 0) {
                if (w) atomicAdd((unsigned long long*)&work[r], w);
                acc.w += w;
                if (wp == 0) acc.add((unsigned long long)(e - h), (unsigned long long)(e - b), 0);
            }
        }
    }
    const int64_t first = list ? 0 : row_ptr[b1], last = list ? 0 : row_ptr[n];
    for (int64_t x0 = first + w0 * kRowSegment; x0 < last; x0 += warps * kRowSegment) {
        const int64_t x1 = x0 + kRowSegment < last ? x0 + kRowSegment : last;
        // row of position x0: the last one that starts at or before it
        int64_t lo = b1, hi = n;
        while (hi - lo > 1) {
            const int64_t step = (hi - lo + 31) >> 5, x = lo + lane * step;
            const unsigned m = __ballot_sync(0xffffffffu, x < hi && row_ptr[x] <= x0) | 1u;
            lo += (31 - __clz(m)) * step;
            hi = hi < lo + step ? hi : lo + step;
        }
        for (int64_t r = lo; r < n; ++r) {
            const int64_t b = row_ptr[r], h = hstart[r], e = row_ptr[r + 1];
            if (b >= x1) break;
            const int64_t q1 = h < x1 ? h : x1;
            unsigned long long w = 0;
#pragma unroll 4
            for (int64_t p = (b > x0 ? b : x0) + lane; p < q1; p += 32) w += (unsigned long long)head[p].hrem;
            w = warp_sum64(w);
            if (lane == 0) {
                if (w) atomicAdd((unsigned long long*)&work[r], w);
                acc.w += w;
                if (b >= x0) acc.add((unsigned long long)(e - h), (unsigned long long)(e - b), 0);
            }
        }
    }
    for (int64_t k = w0; k < mids; k += warps) {
        const int64_t r = list ? list[k] : b1 - 1 - k;
        const int64_t b = row_ptr[r], h = hstart[r], e = row_ptr[r + 1];
        unsigned long long w = 0;
#pragma unroll 4
        for (int64_t p = b + lane; p < h; p += 32) w += (unsigned long long)head[p].hrem;
        w = warp_sum64(w);
        if (lane == 0) {
            work[r] = (int64_t)w;
            acc.add((unsigned long long)(e - h), (unsigned long long)(e - b), w);
        }
    }
    GRID_STRIDE(r, smalls) {
        const int64_t b = row_ptr[r], h = hstart[r], e = row_ptr[r + 1];
        if (e - b > 32) continue;   // a union's mid or hub row
        unsigned long long w = 0;
        for (int64_t p = b; p < h; ++p) w += (unsigned long long)head[p].hrem;
        work[r] = (int64_t)w;
        acc.add((unsigned long long)(e - h), (unsigned long long)(e - b), w);
    }
    for (int o = 16; o; o >>= 1) {
        row_acc x;
        x.h2 = __shfl_xor_sync(0xffffffffu, acc.h2, o);
        x.w = __shfl_xor_sync(0xffffffffu, acc.w, o);
        x.dh = __shfl_xor_sync(0xffffffffu, acc.dh, o);
        x.maxh = __shfl_xor_sync(0xffffffffu, acc.maxh, o);
        x.maxd = __shfl_xor_sync(0xffffffffu, acc.maxd, o);
        acc.join(x);
    }
    if (lane == 0) s_acc[wp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < kRowWarps; ++k) acc.join(s_acc[k]);
        if (acc.maxd) {   // some row with entries
            atomicAdd(&st->sum_h2, acc.h2);
            atomicAdd(&st->wedges, acc.w);
            atomicAdd(&st->sum_dh, acc.dh);
            atomicMax(&st->max_h, acc.maxh);
            atomicMax(&st->max_d, acc.maxd);
        }
    }
}

int bits_for(int64_t n) {
    int b = 1;
    while (b < 62 && ((int64_t)1 << b) < n) ++b;
    return b;
}

// Owns every temporary of a build so that an early return releases them.
struct scratch {
    cudaStream_t s;
    std::vector<void*> p;
    explicit scratch(cudaStream_t st) : s(st) { p.reserve(64); }
    template <typename T>
    tc_status get(T** out, size_t count) {
        void* q = nullptr;
        *out = nullptr;
        TC_TRY(dalloc(&q, count * sizeof(T) + 16, s));
        p.push_back(q);
        *out = (T*)q;
        return TC_OK;
    }
    ~scratch() {
        for (void* q : p) dfree(q, s);
    }
};

template <typename T>
tc_status sort_keys(scratch& sc, cub::DoubleBuffer<T>& buf, int64_t count, int end_bit, cudaStream_t s) {
    size_t bytes = 0;
    TC_CUDA(cub::DeviceRadixSort::SortKeys(nullptr, bytes, buf, count, 0, end_bit, s));
    uint8_t* tmp = nullptr;
    TC_TRY(sc.get(&tmp, bytes));
    // called inside a launch_scope: the sort's own kernels counted beyond it
    const int64_t k = library_kernels("radix_sort_keys", count, end_bit, [&](cudaStream_t p) {
        cub::DoubleBuffer<T> probe = buf;   // the real call flips buf's selector
        return cub::DeviceRadixSort::SortKeys(tmp, bytes, probe, count, 0, end_bit, p);
    });
    TC_CUDA(cub::DeviceRadixSort::SortKeys(tmp, bytes, buf, count, 0, end_bit, s));
    add_launches(k - 1);
    return TC_OK;
}

tc_status sort_by_key(scratch& sc, cub::DoubleBuffer<uint32_t>& keys, cub::DoubleBuffer<int32_t>& vals, int64_t count,
                      int end_bit, cudaStream_t s) {
    size_t bytes = 0;
    TC_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, bytes, keys, vals, count, 0, end_bit, s));
    uint8_t* tmp = nullptr;
    TC_TRY(sc.get(&tmp, bytes));
    const int64_t k = library_kernels("radix_sort_pairs", count, end_bit, [&](cudaStream_t p) {
        cub::DoubleBuffer<uint32_t> kp = keys;   // the real call flips the selectors
        cub::DoubleBuffer<int32_t> vp = vals;
        return cub::DeviceRadixSort::SortPairs(tmp, bytes, kp, vp, count, 0, end_bit, p);
    });
    TC_CUDA(cub::DeviceRadixSort::SortPairs(tmp, bytes, keys, vals, count, 0, end_bit, s));
    add_launches(k - 1);
    return TC_OK;
}

// Step 4 after the run offsets: row split and cursors, tail placement,
// then the runs sorted and written by length class.
template <class C>
tc_status build_runs(tc_graph* g, cudaStream_t s, int64_t m, int64_t n, int bits, const uint64_t* keys,
                     uint64_t* slot, const int32_t* dh, const int64_t* hptr, int32_t* big, unsigned int* nbig,
                     C* hnext, C* tnext, int64_t core_t) {
    {
        launch_scope ls("build_hstart", s);
        k_hstart<<<grid_for(n), kThreads, 0, s>>>(g->row_ptr, dh, hptr, n, g->hstart, hnext, tnext, g->work);
        TC_LAUNCH_CHECK();
    }
    {
        launch_scope ls("build_tail_place", s);
        k_tail_place<<<ordered_blocks(m, kThreads * kPlace), kThreads, 0, s>>>(keys, m, bits, tnext, slot);
        TC_LAUNCH_CHECK();
    }
    {
        launch_scope ls("build_runs_small", s);
        const int rows = n < (int64_t)sm_count() * kSmallRowsFrom ? 4 : 32;
        const int64_t warps = (n + rows - 1) / rows, per = rows == 32 ? kThreads / 32 : 1;
        k_runs_small<<<ordered_blocks(warps, per), (int)(32 * per), 0, s>>>(
            g->row_ptr, g->hstart, hptr, slot, n, hnext, g->col, g->head, (C*)g->edge_tail, big, nbig, core_t, rows);
        TC_LAUNCH_CHECK();
    }
    {
        launch_scope ls("build_runs_mid", s);
        if (TC_RUNS_REG)
            k_runs_mid_reg<C><<<sm_count() * 16, 32 * kMidWarps, 0, s>>>(
                g->row_ptr, g->hstart, hptr, slot, big, nbig, hnext, g->col, g->head, (C*)g->edge_tail, core_t);
        else
            k_runs_mid<C, kMidShort><<<sm_count() * 16, 32 * kMidWarps, 0, s>>>(
                g->row_ptr, g->hstart, hptr, slot, big, nbig, n, hnext, g->col, g->head, (C*)g->edge_tail, core_t);
        TC_LAUNCH_CHECK();
    }
    {
        launch_scope ls("build_runs_long", s);
        if (TC_RUNS_CTA_REG)
            k_runs_long_cta<C><<<sm_count() * 16, 32 * kMidWarps, 0, s>>>(
                g->row_ptr, g->hstart, hptr, slot, big, nbig, n, hnext, g->col, g->head, (C*)g->edge_tail, core_t);
        else
            k_runs_mid<C, kMidRun><<<sm_count() * 8, 32 * kMidWarps, 0, s>>>(
                g->row_ptr, g->hstart, hptr, slot, big, nbig, n, hnext, g->col, g->head, (C*)g->edge_tail, core_t);
        TC_LAUNCH_CHECK();
    }
    {
        launch_scope ls("build_runs_big", s);
        k_runs_big<<<sm_count() * 2, kRunThreads, 0, s>>>(g->row_ptr, g->hstart, hptr, slot, big, nbig, n,
                                                          hnext, g->col, g->head, (C*)g->edge_tail, core_t);
        TC_LAUNCH_CHECK();
    }
    return TC_OK;
}

}  // namespace

void free_graph_memory(tc_graph* g) {
    cudaStream_t s = g->stream;
    void* ptrs[] = {g->edge_u, g->edge_v, g->perm, g->row_ptr, g->col, g->hstart, g->head,
                    g->edge_tail, g->work, g->tri, g->flag, g->tri32, g->counters, g->ecnt, g->row_list};
    for (void* q : ptrs) dfree(q, s);
    free_plan(g->plan, s);
}

tc_status build_graph(tc_graph* g, const void* src, const void* dst, int64_t np, int64_t n,
                      uint32_t flags, cudaStream_t s, const union_layout* un) {
    g->n = n;
    g->bits = bits_for(n);
    g->stream = s;
    const int bits = g->bits;
    const int low_bits = un ? bits_for(un->max_n) : bits;   // low part of a canonical key
    const bool i32 = (flags & TC_IDS_INT32) != 0;
    const size_t id_bytes = i32 ? 4 : 8;
    scratch sc(s);

    // ---- 0. inputs on the device
    const void* dsrc = src;
    const void* ddst = dst;
    if (!(flags & TC_IN_DEVICE) && np > 0) {
        void *a = nullptr, *b = nullptr;
        TC_TRY(sc.get((uint8_t**)&a, np * id_bytes));
        TC_TRY(sc.get((uint8_t**)&b, np * id_bytes));
        copy_scope cs("copy_h2d_pairs", s);
        TC_CUDA(cudaMemcpyAsync(a, src, np * id_bytes, cudaMemcpyHostToDevice, s));
        TC_CUDA(cudaMemcpyAsync(b, dst, np * id_bytes, cudaMemcpyHostToDevice, s));
        dsrc = a;
        ddst = b;
    }

    // ---- 1-2. canonical undirected edges
    unsigned int* err = nullptr;
    TC_TRY(sc.get(&err, 4));
    TC_CUDA(cudaMemsetAsync(err, 0, 4, s));
    uint64_t *ka = nullptr, *kb = nullptr;
    int64_t m = 0;
    int64_t* d_nsel = nullptr;
    TC_TRY(sc.get(&d_nsel, 2));
    if (np > 0) {
        TC_TRY(sc.get(&ka, np));
        TC_TRY(sc.get(&kb, np));
        const int key_bits = bits + low_bits;
        const bool msd = np >= kMsdPairs && np < ((int64_t)1 << 32);   // 32-bit counts in the sort
        digit_counts dc{};
        if (msd) {
            const int d0 = sort_first_digit(np, key_bits);
            dc.bins = 1 << d0;
            dc.shift = key_bits - d0;
            TC_TRY(sc.get(&dc.cnt, dc.bins));
            TC_CUDA(cudaMemsetAsync(dc.cnt, 0, dc.bins * 4, s));
        }
        {
            launch_scope ls("build_make_keys", s);
            if (un && i32)
                k_make_union_keys<int32_t><<<grid_for(np, 8), kThreads, 0, s>>>(
                    (const int32_t*)dsrc, (const int32_t*)ddst, np, *un, low_bits, ka, err, dc);
            else if (un)
                k_make_union_keys<int64_t><<<grid_for(np, 8), kThreads, 0, s>>>(
                    (const int64_t*)dsrc, (const int64_t*)ddst, np, *un, low_bits, ka, err, dc);
            else if (i32)
                k_make_keys<int32_t><<<grid_for(np), kThreads, 0, s>>>(
                    (const int32_t*)dsrc, (const int32_t*)ddst, np, n, bits, ka, err, dc);
            else
                k_make_keys<int64_t><<<grid_for(np), kThreads, 0, s>>>(
                    (const int64_t*)dsrc, (const int64_t*)ddst, np, n, bits, ka, err, dc);
            TC_LAUNCH_CHECK();
        }
        uint64_t *sorted = nullptr, *uniq = nullptr;
        int64_t count = np;
        if (msd) {
            TC_TRY(sort_keys_msd([&](void** q, size_t bytes) { return sc.get((uint8_t**)q, bytes); }, ka, kb, dc.cnt,
                                 np, key_bits, err, &sorted, &count, s));
            uniq = sorted == ka ? kb : ka;
        } else {
            cub::DoubleBuffer<uint64_t> kbuf(ka, kb);
            launch_scope ls("build_sort_pairs", s);
            TC_TRY(sort_keys(sc, kbuf, np, key_bits, s));
            sorted = kbuf.Current();
            uniq = kbuf.Alternate();
        }
        if (count > 0) {
            size_t bytes = 0;
            TC_CUDA(cub::DeviceSelect::Unique(nullptr, bytes, sorted, uniq, d_nsel, count, s));
            uint8_t* tmp = nullptr;
            TC_TRY(sc.get(&tmp, bytes));
            {
                launch_scope ls("build_unique", s);
                TC_TRY(run_library("select_unique", np, 0, true, s, [&](cudaStream_t st) {
                    return cub::DeviceSelect::Unique(tmp, bytes, sorted, uniq, d_nsel, count, st);
                }));
            }
            {
                launch_scope ls("build_edge_count", s);
                k_edge_count<<<1, 1, 0, s>>>(uniq, err, d_nsel);
                TC_LAUNCH_CHECK();
            }
            int64_t got[2] = {0, 0};
            TC_CUDA(cudaMemcpyAsync(got, d_nsel, sizeof(got), cudaMemcpyDeviceToHost, s));
            TC_CUDA(cudaStreamSynchronize(s));
            if (got[1]) return TC_ERR_INVALID_ARG;
            m = got[0];
        }
        ka = uniq;  // the m unique keys
    }
    if (m >= ((int64_t)1 << 32)) return TC_ERR_INVALID_ARG;  // edge ids are 32-bit
    g->m = m;
    const int64_t e2 = 2 * m;

    // ---- graph-owned arrays
    TC_TRY(dalloc((void**)&g->edge_u, (m + 1) * 4, s));
    TC_TRY(dalloc((void**)&g->edge_v, (m + 1) * 4, s));
    TC_TRY(dalloc((void**)&g->perm, (n + 1) * 4, s));
    TC_TRY(dalloc((void**)&g->row_ptr, (n + 2) * 8, s));
    // 32 ids of padding: the count step reads whole groups of 16-byte
    // units, and the last group of the last row may extend past 2m
    TC_TRY(dalloc((void**)&g->col, (e2 + 32) * 4, s));
    TC_CUDA(cudaMemsetAsync(g->col + e2, 0xff, 32 * 4, s));
    TC_TRY(dalloc((void**)&g->hstart, (n + 1) * 8, s));
    TC_TRY(dalloc((void**)&g->head, (e2 + 1) * sizeof(tc_head), s));
    TC_TRY(dalloc(&g->edge_tail, (m + 1) * (g->narrow() ? 4 : 8), s));
    TC_TRY(dalloc((void**)&g->work, (n + 1) * 8, s));
    TC_TRY(dalloc((void**)&g->tri, (n + 1) * 8, s));
    TC_TRY(dalloc((void**)&g->tri32, (n + 1) * 4, s));
    TC_TRY(dalloc((void**)&g->flag, flag_words(e2) * 4, s));
    TC_TRY(dalloc((void**)&g->counters, 8 * 8, s));

    // ---- 3. degrees and the order π
    int32_t* deg = nullptr;
    TC_TRY(sc.get(&deg, n + 1));
    TC_CUDA(cudaMemsetAsync(deg, 0, (n + 1) * 4, s));
    if (m > 0) {
        launch_scope ls("build_edges_degrees", s);
        k_edges_degrees<<<ordered_blocks(m, kThreads), kThreads, 0, s>>>(ka, m, low_bits, un != nullptr, g->edge_u, g->edge_v,
                                                         deg);
        TC_LAUNCH_CHECK();
    }
    int32_t* rank = nullptr;
    int64_t *degr = nullptr, *d_band = nullptr;
    TC_TRY(sc.get(&d_band, 2));
    TC_TRY(sc.get(&rank, n + 1));
    TC_TRY(sc.get(&degr, n + 2));
    if (n > 0) {
        uint32_t *ra = nullptr, *rb = nullptr;
        int32_t *la = nullptr, *lb = nullptr, *lg = nullptr;
        TC_TRY(sc.get(&ra, n));
        TC_TRY(sc.get(&rb, n));
        TC_TRY(sc.get(&la, n));
        TC_TRY(sc.get(&lb, n));
        if (un) {
            // at most 2m / 33 rows of degree above 32, 2m / 4097 hubs
            g->hub_at = e2 / 33 + 1;
            TC_TRY(dalloc((void**)&g->row_list, (g->hub_at + e2 / (TC_BAND_CTA + 1) + 1) * 4, s));
            TC_TRY(sc.get(&lg, n));
            launch_scope ls("build_label_graph", s);
            k_label_graph<<<grid_for(n, 8), kThreads, 0, s>>>(*un, n, lg);
            TC_LAUNCH_CHECK();
        }
        // the key needs as many degree bits as the largest degree has: read
        // back where a sort pass (8 bits) costs more than the wait for it,
        // else bounded by the vertices of a graph and by m
        rank_key rk{};
        rk.dbits = bits_for(std::min((un ? un->max_n : n) - 1, m) + 1);
        if (n > kMaxDegreeReadBack) {
            int32_t* d_maxdeg = nullptr;
            TC_TRY(sc.get(&d_maxdeg, 1));
            TC_CUDA(cudaMemsetAsync(d_maxdeg, 0, 4, s));
            {
                launch_scope ls("build_max_degree", s);
                k_max_degree<<<grid_for(n, 8), kThreads, 0, s>>>(deg, n, d_maxdeg);
                TC_LAUNCH_CHECK();
            }
            int32_t maxdeg = 0;
            TC_CUDA(cudaMemcpyAsync(&maxdeg, d_maxdeg, 4, cudaMemcpyDeviceToHost, s));
            TC_CUDA(cudaStreamSynchronize(s));
            rk.dbits = bits_for((int64_t)maxdeg + 1);
        }
        if (un && un->G > 1) {
            rk.gbits = bits_for(un->G);
            if (rk.dbits + rk.gbits > 32) {   // dbits <= 31
                rk.gshift = std::min(rk.gbits, rk.dbits + rk.gbits - 32);
                rk.gbits -= rk.gshift;
            }
        }
        {
            launch_scope ls("build_rank_keys", s);
            k_rank_keys<<<grid_for(n), kThreads, 0, s>>>(deg, n, rk, lg, ra, la, d_band);
            TC_LAUNCH_CHECK();
        }
        cub::DoubleBuffer<uint32_t> rbuf(ra, rb);
        cub::DoubleBuffer<int32_t> lbuf(la, lb);
        {
            launch_scope ls("build_sort_rank", s);
            TC_TRY(sort_by_key(sc, rbuf, lbuf, n, rk.dbits + rk.gbits, s));
        }
        launch_scope ls("build_rank_apply", s);
        k_rank_apply<<<ordered_blocks(n, kThreads), kThreads, 0, s>>>(rbuf.Current(), lbuf.Current(), n, rk.dbits, lg, g->perm, rank,
                                                      degr, un ? un->rank_graph : nullptr, d_band, g->row_list,
                                                      g->hub_at);
        TC_LAUNCH_CHECK();
    } else {
        TC_CUDA(cudaMemsetAsync(degr, 0, 8, s));
        TC_CUDA(cudaMemsetAsync(d_band, 0, 2 * 8, s));
    }
    {
        size_t bytes = 0;
        TC_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, bytes, degr, g->row_ptr, n + 1, s));
        uint8_t* tmp = nullptr;
        TC_TRY(sc.get(&tmp, bytes));
        launch_scope ls("build_row_ptr", s);
        TC_TRY(run_library("scan_i64", n + 1, 0, true, s, [&](cudaStream_t st) {
            return cub::DeviceScan::ExclusiveSum(tmp, bytes, degr, g->row_ptr, n + 1, st);
        }));
    }

    // ---- 4. rank-space CSR: every edge placed in its lower end's run of
    // tails, each run sorted (N_H(r) ascending) and both entries written;
    // the heads N_L(r) need no order
    if (m > 0) {
        uint64_t *keys = nullptr, *slot = nullptr;
        int32_t *dh = nullptr, *big = nullptr;
        unsigned int* nbig = nullptr;
        void* hnext = nullptr;   // head cursors (absolute positions)
        void* tnext = nullptr;   // tail-run cursors (compact order)
        int64_t* hptr = nullptr;
        TC_TRY(sc.get(&keys, m));
        TC_TRY(sc.get(&slot, m));
        TC_TRY(sc.get(&dh, n + 1));
        TC_TRY(sc.get(&big, n + m / kMidRun + 2));
        TC_TRY(sc.get(&nbig, 3));
        TC_TRY(sc.get((uint8_t**)&hnext, (n + 1) * (g->narrow() ? 4 : 8)));
        TC_TRY(sc.get((uint8_t**)&tnext, (n + 1) * (g->narrow() ? 4 : 8)));
        TC_TRY(sc.get(&hptr, n + 1));
        TC_CUDA(cudaMemsetAsync(dh, 0, (n + 1) * 4, s));
        TC_CUDA(cudaMemsetAsync(nbig, 0, 3 * sizeof(unsigned int), s));
        {
            // in order where a graph's ranks are neighbours (the 8192-graph batch:
            // 2.45 -> 1.78 ms); in a single graph neighbouring edges then add to
            // the same few counters at once (R-MAT scale 24: 2.6 -> 4.1)
            launch_scope ls("build_edge_rank_keys", s);
            k_edge_rank_keys<<<un ? ordered_blocks(m, kThreads) : grid_for(m), kThreads, 0, s>>>(g->edge_u, g->edge_v, rank, m, bits, keys, dh);
            TC_LAUNCH_CHECK();
        }
        size_t sbytes = 0;
        TC_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, sbytes, dh, hptr, n + 1, s));
        uint8_t* tmp = nullptr;
        TC_TRY(sc.get(&tmp, sbytes));
        {
            launch_scope ls("build_hptr", s);
            TC_TRY(run_library("scan_i32", n + 1, 0, true, s, [&](cudaStream_t st) {
                return cub::DeviceScan::ExclusiveSum(tmp, sbytes, dh, hptr, n + 1, st);
            }));
        }
        // the dense core, if one pays: its rows' head records stream nothing
        TC_TRY(core_setup(g, dh, flags, s));
        const int64_t core_t = n - g->core_c;
        if (g->narrow()) {
            TC_TRY(build_runs(g, s, m, n, bits, keys, slot, dh, hptr, big, nbig, (uint32_t*)hnext,
                              (uint32_t*)tnext, core_t));
        } else {
            TC_TRY(build_runs(g, s, m, n, bits, keys, slot, dh, hptr, big, nbig, (unsigned long long*)hnext,
                              (unsigned long long*)tnext, core_t));
        }
    } else if (n > 0) {
        // no edges: every row is empty
        TC_CUDA(cudaMemsetAsync(g->hstart, 0, n * 8, s));
    }

    // ---- 6. per-row work, statistics and the count-step plan
    row_stats* dst_stats = nullptr;
    TC_TRY(sc.get(&dst_stats, 1));
    TC_CUDA(cudaMemsetAsync(dst_stats, 0, sizeof(row_stats), s));
    if (n > 0) {
        launch_scope ls("build_row_work", s);
        const int blocks = (int)std::min<int64_t>((n + kRowWarps - 1) / kRowWarps, (int64_t)sm_count() * 8);
        k_row_work<<<blocks, kThreads, 0, s>>>(g->row_ptr, g->hstart, g->head, d_band, g->row_list, g->hub_at, n,
                                               g->work, dst_stats);
        TC_LAUNCH_CHECK();
    }
    row_stats hst{};
    TC_CUDA(cudaMemcpyAsync(&hst, dst_stats, sizeof(row_stats), cudaMemcpyDeviceToHost, s));
    TC_CUDA(cudaMemcpyAsync(g->band, d_band, sizeof(g->band), cudaMemcpyDeviceToHost, s));
    TC_CUDA(cudaStreamSynchronize(s));
    tc_graph_stats& S = g->stats;
    S.n = n;
    S.m = m;
    S.max_degree = (int64_t)hst.max_d;
    S.max_out_degree = (int64_t)hst.max_h;
    S.sum_out_degree_sq = (double)hst.sum_h2;
    S.wedges = (double)hst.wedges;
    S.avg_degeneracy = m ? (double)hst.sum_dh / (double)m : 0.0;
    // the count kernels keep stream lengths and staged indices in 16 bits;
    // |N_H(v)| <= sqrt(2m) makes this reachable only with m >= 2^31 edges
    if (S.max_out_degree >= 65536) return TC_ERR_INVALID_ARG;
    // Count step: stage N_H(v) once per middle vertex (4m), read each head
    // entry's label, twin and stream length (16m), stream every wedge id
    // (4 W), write the vertex counts (8n) and one flag byte per tail entry (m).
    S.count_bytes = 4.0 * m + 16.0 * m + 4.0 * S.wedges + 8.0 * n + 1.0 * m;
    // Gather: per vertex row_ptr, hstart, perm, △(v), numerator and TC out
    // (8+8+4+8+8+8) and the 32-bit copy of △(v) made first (8 in, 4 out); per
    // adjacency entry its label and the neighbour's count from that copy
    // (4+4); per head entry twin and the mirrored flag (8+1); per tail entry
    // its flag (1).
    S.centrality_bytes = 56.0 * n + 8.0 * (double)e2 + 9.0 * m + 1.0 * m;
    // Target work of a CTA item: large items stage N_H(v) less often, small
    // ones spread a few heavy vertices over more CTAs.  About 64 items' worth
    // of the graph's wedges per SM, within [2^16, 2^22] (R-MAT scale 24: 2^22;
    // the 4096^2 grid with its Chung-Lu hubs: 2^16, where 2^22 left the
    // bitmap kernel 2.5 times slower).  tc_set_plan_params overrides it.
    {
        const double per = S.wedges / (64.0 * (double)sm_count());
        g->params.cta_chunk = (int64_t)std::min(4194304.0, std::max(65536.0, per));
        // Of few wedges, the longest warp items, of up to 4096, set the count's
        // time: smaller ones, by the same measure (a count: R-MAT scale 12 98 ->
        // 74 us, 16 274 -> 174, 300^2 grid 203 -> 83, 600^2 grid 482 -> 145).
        // With more every warp has several and the staging counts: R-MAT
        // scale 17, at 9000 a warp's share, 256 us, 272 in items of 512.
        if (per < 4096.0) g->params.warp_split = (int64_t)std::min(512.0, std::max(128.0, per));
    }
    // Unions of many small graphs hold millions of light vertices; one
    // thread each for those of up to 128 ids of work instead of 64 (the
    // 8192-graph batch: count 7.9 -> 6.7 ms; on the grid workload the
    // larger cap was 0.3 ms slower, so single graphs keep 64).  With fewer
    // vertices the longest thread items set that kernel's time: 64 where a
    // thread has few (a union of 500 graphs, 1.6 M vertices: a run 0.345 ->
    // 0.315 ms; caps of 32 and 16 0.356 and 0.438), 16 where the vertices do
    // not keep every thread of the device busy.
    if (n < (int64_t)sm_count() * 2048 * 4) g->params.thread_work = 16;
    else if ((flags & TC_BUILD_NO_CORE) && n >= ((int64_t)1 << 24)) g->params.thread_work = 128;
    TC_TRY(make_plan(g, g->strategy, s));
    TC_CUDA(cudaStreamSynchronize(s));
    return TC_OK;
}

}  // namespace tcx
