// tc_csr_centrality_noalloc: triangle counts, exact numerators and TC for a
// small graph handed over as a device CSR, with every piece of working
// memory taken from one fixed array compiled into this library.
//
// The other entry points draw their working memory (CSR copies, plans, sort
// buffers) from a stream-ordered device pool.  Some callers cannot let a
// library do that: a runtime that owns all device memory through its own
// allocator and forbids hidden allocations, a latency-critical loop where a
// pool growth would stall the device, or a program whose footprint must be
// fixed before it starts.  This variant serves them for graphs up to the
// sizes stated in tc.h.  It computes the same quantities as tc_count
// followed by tc_centrality (Definition 1 through the numerator
// numer(v) = △(v) + Σ_{u∈N(v)} (u ∈ N△(v) ? 1 : 3)·△(u) of Algorithm 2 and
// one division by 3△(G)), with simpler kernels: for every edge the number of
// triangles on it, T(v, u) = |N(v) ∩ N(u)| (T = A² ∘ A, section "Notation"),
// by testing the shorter of the two rows against a bitmap of the longer one;
// then △(v) = ½ Σ_u T(v, u), △(G) = ⅓ Σ_edges T and the edge's flag is T > 0.
#include <algorithm>
#include <mutex>

#include "tc_internal.cuh"

namespace {

typedef unsigned long long ull;

constexpr int64_t kMaxN = TC_NOALLOC_MAX_VERTICES;
constexpr int64_t kMaxNnz = TC_NOALLOC_MAX_ENTRIES;
constexpr int64_t kFlagWords = kMaxNnz / 64;          // one bit per CSR entry
constexpr int64_t kTriOff = 0;                        // 2△(v), kMaxN words
constexpr int64_t kFlagOff = kTriOff + kMaxN;         // edge flags, kFlagWords words
constexpr int64_t kDenOff = kFlagOff + kFlagWords;    // Σ_v △(v) = 3△(G)
constexpr int64_t kErrOff = kDenOff + 1;              // nonzero: the input broke a rule
constexpr int64_t kFoundOff = kErrOff + 1;            // edges whose two entries were both seen
constexpr int64_t kWords = (kFoundOff + 1 + 31) / 32 * 32;   // 786,688 bytes

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int64_t kBigRow = 256;   // rows above it take a whole CTA in the gather

}  // namespace

// The whole working set, 768 KB per device, allocated when the module is
// loaded.  Every word a call uses (counts, flags, 3△(G), error word) is
// cleared by k_na_clear at the start of that call, so nothing carries over
// from one call to the next.
static __device__ __align__(256) unsigned long long g_noalloc_scratch[kWords];

namespace {

struct na_args;
__global__ void k_na_count(na_args a, int per);
__host__ __device__ size_t na_count_smem(int64_t n);

// Device address of g_noalloc_scratch per device, looked up once.
constexpr int kMaxDevices = 64;
std::mutex g_setup_mu;
ull* g_scratch_ptr[kMaxDevices] = {};

tc_status scratch_for_current_device(ull** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return tcx::from_cuda(e);
    if (dev < 0 || dev >= kMaxDevices) return TC_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return tcx::from_cuda(e);
        if (!p) return TC_ERR_CUDA;
        // once per device too, and before any capture: the largest staging
        e = cudaFuncSetAttribute(k_na_count, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)na_count_smem(kMaxN));
        if (e != cudaSuccess) return tcx::from_cuda(e);
        g_scratch_ptr[dev] = (ull*)p;
    }
    *out = g_scratch_ptr[dev];
    return TC_OK;
}

struct na_args {
    const int64_t* row_ptr;
    const int32_t* col;
    int64_t n, nnz;
    ull* tri;
    ull* flag;
    ull* den;
    ull* err;
    ull* found;
};

// Shared words of one warp of k_na_count: a bit per vertex, then per entry
// of its unit the walk's prefix, the row's start, T and the back position.
__host__ __device__ __forceinline__ int na_bitmap_words(int64_t n) { return (int)((((n + 31) >> 5) + 31) & ~31ll); }
__host__ __device__ size_t na_count_smem(int64_t n) {
    return (size_t)kWarps * (na_bitmap_words(n) + 4 * 32) * 4;
}

__device__ __forceinline__ void na_fail(const na_args& a) { atomicOr(a.err, 1ull); }

// Row [b, e) of x, or false (and the error word set) if row_ptr breaks
// 0 = row_ptr[0] <= ... <= row_ptr[n] = nnz at x, or the row has more
// entries than there are other vertices.
__device__ __forceinline__ bool na_row(const na_args& a, int64_t x, int64_t& b, int64_t& e) {
    b = a.row_ptr[x];
    e = a.row_ptr[x + 1];
    bool ok = 0 <= b && b <= e && e <= a.nnz && e - b < a.n && (x != 0 || b == 0) && (x != a.n - 1 || e == a.nnz);
    if (!ok) na_fail(a);
    return ok;
}

__device__ __forceinline__ bool na_flag_get(const na_args& a, int64_t pos) {
    return (a.flag[pos >> 6] >> (pos & 63)) & 1ull;
}

// The input is a simple symmetric CSR: no check failed, and every entry is
// one of the two of an edge that was seen from both ends.
__device__ __forceinline__ bool na_valid(const na_args& a) {
    return *a.err == 0 && 2 * *a.found == (ull)a.nnz;
}

__device__ __forceinline__ ull na_warp_sum(ull x) {
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

__global__ void k_na_clear(ull* scratch, int64_t n, int64_t nnz) {
    tcx::pdl_trigger();
    tcx::pdl_wait();
    const int64_t flag_words = (nnz + 63) / 64;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n + flag_words + 3; i += stride) {
        if (i < n) scratch[kTriOff + i] = 0;
        else if (i < n + flag_words) scratch[kFlagOff + (i - n)] = 0;
        else scratch[kDenOff + (i - n - flag_words)] = 0;   // den, err, found
    }
}

// T(v, u) of every edge, once, from its end v of larger degree (ties: larger
// id).  A warp takes 32 (small graphs: 16) consecutive entries (v, u) at a
// time, one per lane; for each row v among them N(v) becomes a bitmap over all n ids in the
// warp's shared memory (at most 8 KB), and the rows u of the lanes' entries
// are walked as one concatenation, each id one coalesced load and one bit
// test, hits counted in a register until the walk leaves the row.  The walk
// also meets v itself in row u, unless the CSR is not symmetric: that gives
// the position of the edge's other entry, flagged with this one, and the
// count of edges seen from both ends (compared with nnz / 2 at the end).
// The work, Σ_edges min(d_u, d_v) ids, is spread over the entries, so hubs
// are shared by as many warps as they have entries / 32.
// One warp a vertex with a binary search for every pair of later neighbours
// took 6.2 ms on the R-MAT scale-12 graph (47 K edges), nearly all of it in
// the chains of searches of a few hub rows; this takes 30 us there, bound by
// the latency of the longest unit's loads (eight in flight a lane: 37 -> 30
// with four and units of 32), and 0.62 ms on a scale-16 graph near both size
// limits (0.8 M edges, 1.5e8 ids).
__global__ void __launch_bounds__(kThreads) k_na_count(na_args a, int per) {
    tcx::pdl_trigger();
    tcx::pdl_wait();
    extern __shared__ uint32_t na_sh[];
    const int words = na_bitmap_words(a.n);
    const int lane = threadIdx.x & 31;
    uint32_t* bm = na_sh + (threadIdx.x >> 5) * (words + 4 * 32);
    int* s_pre = (int*)(bm + words);
    int* s_base = s_pre + 32;
    int* s_back = s_base + 32;
    uint32_t* s_t = (uint32_t*)(s_back + 32);
    for (int i = lane; i < words; i += 32) bm[i] = 0;
    __syncwarp();
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t threads = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = tid; x < a.n; x += threads) {
        int64_t b, e;
        na_row(a, x, b, e);   // every row's offsets, empty rows too
    }
    const uint32_t n = (uint32_t)a.n;
    ull den = 0, found = 0;
    const int64_t units = (a.nnz + per - 1) / per;
    for (int64_t unit = tid >> 5; unit < units; unit += threads >> 5) {
        const int64_t p0 = unit * per, p = p0 + lane;
        const bool live = lane < per && p < a.nnz;
        // row of the unit's first entry (the last x with row_ptr[x] <= p0),
        // 32 probes at a time; then each lane steps on to its own
        int64_t lo = 0, hi = a.n;
        while (hi - lo > 1) {
            const int64_t step = (hi - lo + 31) >> 5, x = lo + lane * step;
            const unsigned m = __ballot_sync(0xffffffffu, x < hi && a.row_ptr[x] <= p0) | 1u;
            lo += (31 - __clz(m)) * step;
            hi = hi < lo + step ? hi : lo + step;
        }
        int64_t v = lo;
        {
            int64_t step = 1;
            while (v + step < a.n && a.row_ptr[v + step] <= p) {
                v += step;
                step <<= 1;
            }
            while (step > 1) {
                step >>= 1;
                if (v + step < a.n && a.row_ptr[v + step] <= p) v += step;
            }
        }
        int64_t b = 0, e = 0, ub = 0, ue = 0;
        int32_t u = -1;
        bool ok = live && na_row(a, v, b, e);
        if (ok && (p < b || p >= e)) {
            na_fail(a);
            ok = false;
        }
        if (ok) {
            u = a.col[p];
            // ids in range, strictly increasing along the row
            if ((uint32_t)u >= n || (p > b && a.col[p - 1] >= u)) {
                na_fail(a);
                ok = false;
            }
        }
        if (ok) ok = na_row(a, u, ub, ue);
        const bool mine = ok && (ue - ub < e - b || (ue - ub == e - b && u < v));
        unsigned todo = __ballot_sync(0xffffffffu, mine);
        if (!todo) continue;
        s_base[lane] = (int)ub;
        s_back[lane] = -1;
        s_t[lane] = 0;
        while (todo) {
            const int lead = __ffs(todo) - 1;
            const int64_t vv = __shfl_sync(0xffffffffu, v, lead);
            const int64_t vb = __shfl_sync(0xffffffffu, b, lead), ve = __shfl_sync(0xffffffffu, e, lead);
            const bool in = mine && v == vv;
            todo &= ~__ballot_sync(0xffffffffu, in);
#pragma unroll 4
            for (int64_t i = vb + lane; i < ve; i += 32) {
                const uint32_t c = (uint32_t)a.col[i];
                if (c < n) atomicOr(&bm[c >> 5], 1u << (c & 31));
            }
            const int len = in ? (int)(ue - ub) : 0;
            int incl = len;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += x;
            }
            s_pre[lane] = incl - len;
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            __syncwarp();
            constexpr int K = 8;   // independent loads a lane has in flight
            int at = 0, cur = 0;
            uint32_t hits = 0;
            for (int q0 = lane; q0 < total; q0 += 32 * K) {
                int32_t c[K];
                int row[K], pos[K];
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    const int q = q0 + 32 * j;
                    c[j] = -1;
                    row[j] = at;
                    pos[j] = 0;
                    if (q < total) {
                        while (at < 31 && s_pre[at + 1] <= q) ++at;
                        row[j] = at;
                        pos[j] = s_base[at] + q - s_pre[at];
                        c[j] = a.col[pos[j]];
                    }
                }
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    if ((uint32_t)c[j] >= n) continue;
                    if (row[j] != cur) {
                        if (hits) atomicAdd(&s_t[cur], hits);
                        hits = 0;
                        cur = row[j];
                    }
                    hits += (bm[c[j] >> 5] >> (c[j] & 31)) & 1u;
                    if (c[j] == (int32_t)vv) s_back[cur] = pos[j];
                }
            }
            if (hits) atomicAdd(&s_t[cur], hits);
            __syncwarp();
            if (words <= ve - vb) {
                for (int i = lane; i < words; i += 32) bm[i] = 0;
            } else {
                for (int64_t i = vb + lane; i < ve; i += 32) {
                    const uint32_t c = (uint32_t)a.col[i];
                    if (c < n) bm[c >> 5] = 0;
                }
            }
            const uint32_t t = in ? s_t[lane] : 0;
            const int back = in ? s_back[lane] : -1;
            if (back >= 0) ++found;
            const unsigned marked = __ballot_sync(0xffffffffu, t != 0);
            if (t) {
                atomicAdd(a.tri + u, (ull)t);
                if (back >= 0) atomicOr(a.flag + (back >> 6), 1ull << (back & 63));
            }
            const uint32_t sum = __reduce_add_sync(0xffffffffu, t);
            if (lane == lead && sum) {
                atomicAdd(a.tri + vv, (ull)sum);
                // p0 is a multiple of per (16 or 32): the unit's flags lie in one word
                atomicOr(a.flag + (p0 >> 6), (ull)marked << (p0 & 63));
                den += sum;
            }
            __syncwarp();
        }
    }
    den = na_warp_sum(den);
    found = na_warp_sum(found);
    if (lane == 0) {
        if (den) atomicAdd(a.den, den);   // Σ_edges T = 3△(G)
        if (found) atomicAdd(a.found, found);
    }
}

__device__ __forceinline__ void na_finish(const na_args& a, int64_t v, ull acc, ull den, ull* d_tri, ull* d_numer,
                                          double* d_tc) {
    const ull t = a.tri[v] >> 1;
    acc += t;
    if (d_tri) d_tri[v] = t;
    if (d_numer) d_numer[v] = acc;
    if (d_tc)
        d_tc[v] = den == 0 ? __longlong_as_double(0x7ff8000000000000ll) : __ddiv_rn((double)acc, (double)den);
}

// numer(v) = △(v) + Σ_{u∈N(v)} (flag ? 1 : 3)·△(u), the flag of either
// entry of an edge at that entry: one warp per vertex, rows of more than
// kBigRow entries by the whole CTA after its warps' short rows.  Then
// TC(v) = numer(v) / 3△(G): both operands stay below 2^53 within the size
// limits, so one IEEE division is correctly rounded.
__global__ void __launch_bounds__(kThreads) k_na_gather(na_args a, ull* d_tri, ull* d_numer, double* d_tc) {
    tcx::pdl_trigger();
    tcx::pdl_wait();
    __shared__ int64_t s_big[kWarps];
    __shared__ ull s_part[kWarps];
    if (!na_valid(a)) return;   // k_na_mark writes the outputs
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const ull den = *a.den;
    auto term = [&](int64_t p) { return (na_flag_get(a, p) ? 1ull : 3ull) * (a.tri[a.col[p]] >> 1); };
    for (int64_t base = (int64_t)blockIdx.x * kWarps; base < a.n; base += (int64_t)gridDim.x * kWarps) {
        const int64_t v = base + warp;
        int64_t b = 0, e = 0;
        if (v < a.n) {
            b = a.row_ptr[v];
            e = a.row_ptr[v + 1];
        }
        const bool big = e - b > kBigRow;
        if (lane == 0) s_big[warp] = big ? v : -1;
        if (!big) {
            ull acc = 0;
#pragma unroll 4
            for (int64_t p = b + lane; p < e; p += 32) acc += term(p);
            acc = na_warp_sum(acc);
            if (lane == 0 && v < a.n) na_finish(a, v, acc, den, d_tri, d_numer, d_tc);
        }
        __syncthreads();
        for (int k = 0; k < kWarps; ++k) {
            const int64_t w = s_big[k];
            if (w < 0) continue;
            const int64_t wb = a.row_ptr[w], we = a.row_ptr[w + 1];
            ull acc = 0;
#pragma unroll 4
            for (int64_t p = wb + threadIdx.x; p < we; p += kThreads) acc += term(p);
            acc = na_warp_sum(acc);
            if (lane == 0) s_part[warp] = acc;
            __syncthreads();
            if (threadIdx.x == 0) {
                ull sum = 0;
                for (int j = 0; j < kWarps; ++j) sum += s_part[j];
                na_finish(a, w, sum, den, d_tri, d_numer, d_tc);
            }
            __syncthreads();
        }
        __syncthreads();   // s_big is rewritten next
    }
}

// If any check failed, every output is overwritten with its error marker.
__global__ void k_na_mark(na_args a, ull* d_tri, ull* d_numer, double* d_tc) {
    tcx::pdl_trigger();
    tcx::pdl_wait();
    if (na_valid(a)) return;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
        if (d_tri) d_tri[i] = ~0ull;
        if (d_numer) d_numer[i] = ~0ull;
        if (d_tc) d_tc[i] = __longlong_as_double(0x7ff8000000000000ll);
    }
}

}  // namespace

extern "C" tc_status tc_csr_centrality_noalloc(const int64_t* d_row_ptr, const int32_t* d_col, int64_t n,
                                               int64_t nnz, uint64_t* d_tri, uint64_t* d_numer,
                                               double* d_tc, tc_stream stream) {
    tcx::nvtx_range nr("tc_csr_centrality_noalloc");
    if (n < 0 || n > kMaxN || nnz < 0 || nnz > kMaxNnz || (nnz & 1)) return TC_ERR_INVALID_ARG;
    if (n == 0 && nnz != 0) return TC_ERR_INVALID_ARG;
    if (n > 0 && !d_row_ptr) return TC_ERR_INVALID_ARG;
    if (nnz > 0 && !d_col) return TC_ERR_INVALID_ARG;
    ull* scratch = nullptr;
    TC_TRY(scratch_for_current_device(&scratch));
    if (n == 0) return TC_OK;
    cudaStream_t s = (cudaStream_t)stream;
    na_args a{d_row_ptr, d_col, n, nnz, scratch + kTriOff, scratch + kFlagOff, scratch + kDenOff,
              scratch + kErrOff, scratch + kFoundOff};
    const int sms = tcx::sm_count();
    // entries a warp takes at a time: the longest unit's walk sets the time of
    // a small graph, so units are halved where they would leave warps idle
    const int per_entries = nnz < (int64_t)sms * 64 * 32 ? 16 : 32;
    const int64_t units = std::max<int64_t>((nnz + per_entries - 1) / per_entries, (n + 31) / 32);
    const size_t smem = na_count_smem(n);
    const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(8, (size_t)220 * 1024 / (smem + 1024)));
    const int count_blocks = (int)std::min<int64_t>((units + kWarps - 1) / kWarps, (int64_t)sms * per_sm);
    const int row_blocks = (int)std::min<int64_t>((n + kWarps - 1) / kWarps, (int64_t)sms * 8);
    const int flat_blocks = (int)std::min<int64_t>((n + (nnz + 63) / 64 + 3 + 255) / 256, (int64_t)sms * 4);
    TC_CUDA(tcx::launch_pdl(k_na_clear, flat_blocks, 256, 0, s, scratch, n, nnz));
    TC_CUDA(tcx::launch_pdl(k_na_count, count_blocks, kThreads, smem, s, a, per_entries));
    TC_CUDA(tcx::launch_pdl(k_na_gather, row_blocks, kThreads, 0, s, a, (ull*)d_tri, (ull*)d_numer, d_tc));
    TC_CUDA(tcx::launch_pdl(k_na_mark, (int)std::min<int64_t>((n + 255) / 256, (int64_t)sms * 4), 256, 0, s, a,
                            (ull*)d_tri, (ull*)d_numer, d_tc));
    tcx::add_launches(4);
    return TC_OK;
}
