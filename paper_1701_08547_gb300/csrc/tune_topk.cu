// tune_topk: segmented top-k over an external FP32 score array (HBM-bound).
//
// A warp scans its part of a segment in batches of 512 scores (16-byte loads, the next batch in flight
// while the current one is filtered) and keeps an exact list of its 32 best as 64-bit keys
// (order-preserving image of the score, index in the segment), lane j = j-th best. A score is a
// candidate if it does not exceed a bound: first the k-th smallest of the lanes' minima over the first
// batch (k distinct scores do not exceed it), later the list's k-th key. Candidates are only appended to
// a buffer in shared memory; 32 at a time are sorted across the lanes (bitonic) and merged into the
// list. (Inserting them one by one, with the bound taken from the filling list, cost about 37
// insertions of some 60 instructions per 3,000-score segment and was what 20,000 ragged segments spent
// their time on: 92 -> 68 us for 59 M scores with k = 5, 152 -> 62 us with k = 16, the HBM floor being 35.)
// Where many scores are equal, the bound also drops ties as it goes (10,000 segments of 512 equal scores, k = 16: 64 ->
// 25 us), and a batch whose scores are mostly below the bound gets one of its own (1,000 falling sequences of 16,384:
// 348 -> 90 us).
// Short segments have few candidates, which are inserted at their places (k = 1: mostly one), and segments of at most 32
// scores need no batch: 50,000 of 16 scores 43 -> 25 us with k = 1, 53 -> 25 with k = 5; of 200, k = 1, 45 -> 27.
//
// How many warps share a segment (launch()): with more segments than resident CTAs, a warp takes one
// segment after the other; with fewer segments a whole CTA, or a cluster of up
// to eight CTAs, takes one, their lists merged through (distributed) shared memory.
#include <cooperative_groups.h>
#include <stdint.h>

#include "tune_internal.h"

namespace {

namespace cg = cooperative_groups;

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kMaxK = 16;
constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned long long kNone = ~0ull;  // no entry: behind every key
constexpr int kVec = 4;                      // 16-byte loads per lane per batch
constexpr int kBatchF4 = 32 * kVec;          // float4 words per warp batch (2 KB)
constexpr int kInsert = 8;                   // candidates up to which they are inserted one by one
constexpr int kMany = 64;                    // candidates of a batch above which they are taken group by group
constexpr int kLanes = 24;                   // lanes with one above which the batch's own bound is taken again
constexpr float kFltMax = 3.402823466e+38f;

// Monotone map of non-NaN floats to unsigned integers (-inf smallest, +inf largest).
__device__ __forceinline__ unsigned order_key(float f)
{
    unsigned b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ float key_value(unsigned k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// One compare-exchange of a bitonic network: lanes with `lower` keep the smaller of the pair.
template <typename T>
__device__ __forceinline__ T exchange(T x, int mask, bool lower)
{
    const T y = __shfl_xor_sync(kFull, x, mask);
    return (x < y) == lower ? x : y;
}

// Ascending sort across the warp's lanes.
template <typename T>
__device__ __forceinline__ T sort32(T x, int lane)
{
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int m = size >> 1; m > 0; m >>= 1) x = exchange(x, m, ((lane & m) == 0) == ((lane & size) == 0));
    return x;
}

// The 32 smallest of two ascending warp lists, ascending.
__device__ __forceinline__ unsigned long long merge32(unsigned long long a, unsigned long long b, int lane)
{
    const unsigned long long r = __shfl_sync(kFull, b, 31 - lane);
    unsigned long long x = a < r ? a : r;  // bitonic
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) x = exchange(x, m, (lane & m) == 0);
    return x;
}

// v[j] by selects (an index would move the array to local memory).
__device__ __forceinline__ float pick(const float (&v)[4 * kVec], int j)
{
    float t[8], u[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) t[i] = (j & 1) ? v[2 * i + 1] : v[2 * i];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = (j & 2) ? t[2 * i + 1] : t[2 * i];
    const float a = (j & 4) ? u[1] : u[0], b = (j & 4) ? u[3] : u[2];
    return (j & 8) ? b : a;
}

// A segment: `head` scores before the first 16-byte boundary, n4 float4 words, the rest from tail0 on.
struct Segment {
    const float* p;
    int len, head, n4, tail0;
    __device__ __forceinline__ Segment(const float* q, int n) : p(q), len(n)
    {
        head = min((int)(((16u - ((unsigned)reinterpret_cast<uintptr_t>(q) & 15u)) & 15u) >> 2), len);
        n4 = (len - head) >> 2;
        tail0 = head + 4 * n4;
    }
};

// The list and candidate buffer of one warp over its part of a segment.
struct WarpList {
    unsigned long long list;  // this lane's entry, ascending over the lanes
    unsigned long long* buf;  // 64 entries in shared memory, the warp's own
    int cnt, k, lane;
    float thr;  // a score is a candidate if it is <= thr (finite, so neither NaN nor +inf passes)

    __device__ __forceinline__ WarpList(unsigned long long* b, int k_, int l)
        : list(kNone), buf(b), cnt(0), k(k_), lane(l), thr(kFltMax)
    {
    }

    // The first 32 buffered candidates into the list.
    __device__ __forceinline__ void flush()
    {
        __syncwarp();
        if (cnt <= kInsert) {
            for (int i = 0; i < cnt; ++i) insert(buf[i]);
            __syncwarp();
            cnt = 0;
            bound();
            return;
        }
        const unsigned long long x = lane < cnt ? buf[lane] : kNone;
        const unsigned long long more = 32 + lane < cnt ? buf[32 + lane] : kNone;
        __syncwarp();
        if (32 + lane < cnt) buf[lane] = more;
        cnt = max(cnt - 32, 0);
        list = merge32(list, sort32(x, lane), lane);
        bound();
    }

    // One entry, the same on every lane, to its place.
    __device__ __forceinline__ void insert(unsigned long long x)
    {
        const int pos = __popc(__ballot_sync(kFull, list < x));
        const unsigned long long up = __shfl_up_sync(kFull, list, 1);
        list = lane < pos ? list : lane == pos ? x : up;
    }

    // Scores are scanned in increasing index, so once the list holds k entries a later score has to be below the
    // k-th: the bound steps to the next smaller float (past -0, which equals +0).
    __device__ __forceinline__ void bound()
    {
        const unsigned tau = (unsigned)(__shfl_sync(kFull, list, k - 1) >> 32);
        if (tau != 0xffffffffu) {
            const unsigned below = tau == 0x80000000u ? 0x7ffffffeu : tau - 1u;
            thr = tau == 0x007fffffu ? key_value(tau) : fminf(thr, key_value(below));  // -inf: nothing is smaller
        }
    }

    // Every lane with `take` appends one score (all of one stretch of indices above every earlier one);
    // the buffer has room for 32.
    __device__ __forceinline__ void append(bool take, float v, int index)
    {
        const unsigned who = __ballot_sync(kFull, take);
        if (take)  // -0 ranks as +0
            buf[cnt + __popc(who & ((1u << lane) - 1u))] = ((unsigned long long)order_key(v + 0.0f) << 32) | (unsigned)index;
        cnt += __popc(who);
    }

    // Batches first, first + step, ... of the segment's float4 body; with `edges` also its head and tail.
    __device__ __forceinline__ void scan(const Segment& s, int first, int step, bool edges)
    {
        const float nan = __int_as_float(0x7fc00000);
        // the head, or all of a segment of at most 32 scores, one per lane
        const int first_n = s.len <= 32 ? s.len : s.head;
        if (edges && first_n) {
            const float v = lane < first_n ? __ldcs(s.p + lane) : nan;
            append(v <= thr, v, lane);
        }
        if (s.len <= 32) {
            while (cnt > 0) flush();
            return;
        }
        const float4* body = reinterpret_cast<const float4*>(s.p + s.head);
        auto load = [&](float4 (&w)[kVec], int f0) {
#pragma unroll
            for (int q = 0; q < kVec; ++q) {
                const int f = f0 + lane + 32 * q;
                w[q] = f < s.n4 ? __ldcs(body + f) : make_float4(nan, nan, nan, nan);
            }
        };
        float4 cur[kVec];
        int f0 = first * kBatchF4;
        const int df = step * kBatchF4;
        bool fresh = true;
        if (f0 < s.n4) load(cur, f0);
        for (; f0 < s.n4; f0 += df) {
            float v[4 * kVec];
#pragma unroll
            for (int q = 0; q < kVec; ++q) {
                v[4 * q] = cur[q].x;
                v[4 * q + 1] = cur[q].y;
                v[4 * q + 2] = cur[q].z;
                v[4 * q + 3] = cur[q].w;
            }
            if (s.n4 - f0 > df) load(cur, f0 + df);
            float mn = v[0];
#pragma unroll
            for (int j = 1; j < 4 * kVec; ++j) mn = fminf(mn, v[j]);  // fminf skips NaN
            const unsigned who = __ballot_sync(kFull, mn <= thr);
            if (who == 0u) continue;
            if (fresh || __popc(who) > kLanes) {
                // k lanes own a score that does not exceed the k-th smallest of the lanes' minima
                const unsigned key = mn <= kFltMax ? order_key(mn) : 0xffffffffu;
                const unsigned kth = k == 1 ? __reduce_min_sync(kFull, key) : __shfl_sync(kFull, sort32(key, lane), k - 1);
                if (kth != 0xffffffffu) thr = fminf(thr, key_value(kth));
                fresh = false;
            }
            unsigned cm = 0;  // this lane's candidates
#pragma unroll
            for (int j = 0; j < 4 * kVec; ++j) cm |= v[j] <= thr ? 1u << j : 0u;
            // Mostly a candidate per lane at most, and one turn. Many are mostly ties: those are taken float4 group by
            // float4 group (128 consecutive scores), and after each the bound, strict for the higher indices of the
            // groups after it, drops what it excludes.
            unsigned now = __reduce_add_sync(kFull, __popc(cm)) > kMany ? 0xfu : 0xffffu;
            for (;;) {
                const unsigned act = cm & now;
                if (!__any_sync(kFull, act != 0u)) {
                    if (now >= 0xf000u) break;
                    now <<= 4;
                    if (cm & now) {
#pragma unroll
                        for (int j = 0; j < 4 * kVec; ++j) cm &= v[j] <= thr ? ~0u : ~(1u << j);
                    }
                    continue;
                }
                const int j = __ffs(act) - 1;
                append(act != 0u, pick(v, j), s.head + 4 * (f0 + lane + 32 * (j >> 2)) + (j & 3));
                cm &= ~(act & -act);
                if (cnt >= 32) flush();
            }
        }
        if (edges && s.tail0 < s.len) {
            const int i = s.tail0 + lane;
            const float v = i < s.len ? __ldcs(s.p + i) : nan;
            append(v <= thr, v, i);
        }
        while (cnt > 0) flush();
    }

    __device__ __forceinline__ void write(int32_t* out_i, float* out_s) const
    {
        if (lane < k) {
            const unsigned key = (unsigned)(list >> 32);
            out_i[lane] = (int)(unsigned)list;  // -1 for no entry
            out_s[lane] = key == 0xffffffffu ? __int_as_float(0x7f800000) : key_value(key);
        }
    }
};

// The list of a segment whose warps' lists (each its kMaxK best) stand in lists[0..n), on one warp.
__device__ __forceinline__ unsigned long long merge_lists(const unsigned long long (*lists)[kMaxK], int n, int lane)
{
    unsigned long long x = lane < kMaxK ? lists[0][lane] : kNone;
    for (int i = 1; i < n; ++i) x = merge32(x, lane < kMaxK ? lists[i][lane] : kNone, lane);
    return x;
}

// Many segments: CTA b owns per = 2^per_log consecutive ones (2, 4 or 8) of every per x grid; its warps take them one
// after the other from a counter in shared memory, so that a warp with long ones takes fewer. (One queue for the whole
// grid costs 1.5 ns per segment in atomics on one address: 25 us against 15 for 10,000 segments of 64.) The
// next segment's bounds are requested before the current one is scanned. Segments longer than kShare, which
// would keep a warp busy for more than 30 us, are left to the end and shared by the CTA's warps (up to kMaxLong
// of them; 2,400 log-uniform segments of up to 262,144 scores: 300 -> 114 us).
constexpr int kShare = 32768, kMaxLong = 64;
__global__ void __launch_bounds__(kThreads, 4)
    topk_warp_kernel(const float* __restrict__ scores, const int64_t* __restrict__ off, int64_t n_seg, int k,
                     int per_log, int32_t* __restrict__ out_i, float* __restrict__ out_s,
                     unsigned char* __restrict__ header)
{
    static_assert(kThreads == (int)tune::kWorkspaceHeader, "a header byte per thread");
    __shared__ unsigned long long buf[kWarps][64], lists[2][kWarps][kMaxK];
    __shared__ int64_t longs[kMaxLong];
    __shared__ int taken, n_long;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (blockIdx.x == 0) header[threadIdx.x] = 0;  // (no separate launch for that)
    if (threadIdx.x == 0) taken = kWarps, n_long = 0;
    __syncthreads();
    const int per = 1 << per_log;
    auto segment = [&](int i) {
        return (((int64_t)(i >> per_log) * gridDim.x + blockIdx.x) << per_log) + (i & (per - 1));
    };
    int64_t s = segment(warp);
    int64_t b = s < n_seg ? off[s] : 0, e = s < n_seg ? off[s + 1] : 0;
    while (s < n_seg) {
        int i = 0;
        if (lane == 0) i = atomicAdd(&taken, 1);
        const int64_t n = segment(__shfl_sync(kFull, i, 0));
        int64_t nb = 0, ne = 0;
        if (n < n_seg) {
            nb = off[n];
            ne = off[n + 1];
        }
        int slot = kMaxLong;
        if (e - b > kShare) {
            if (lane == 0) slot = atomicAdd(&n_long, 1);
            slot = __shfl_sync(kFull, slot, 0);
        }
        if (slot < kMaxLong) {
            if (lane == 0) longs[slot] = s;
        } else {
            WarpList l(buf[warp], k, lane);
            l.scan(Segment(scores + b, (int)(e - b)), 0, 1, true);
            l.write(out_i + s * k, out_s + s * k);
        }
        s = n;
        b = nb;
        e = ne;
    }
    __syncthreads();
    const int nl = min(n_long, kMaxLong);
    for (int j = 0; j < nl; ++j) {
        const int64_t t = longs[j], tb = off[t];
        WarpList l(buf[warp], k, lane);
        l.scan(Segment(scores + tb, (int)(off[t + 1] - tb)), warp, kWarps, warp == 0);
        if (lane < kMaxK) lists[j & 1][warp][lane] = l.list;
        __syncthreads();
        if (warp == j % kWarps) {  // the other warps go on to the next segment, with the other lists
            l.list = merge_lists(lists[j & 1], kWarps, lane);
            l.write(out_i + t * k, out_s + t * k);
        }
    }
}

// Few segments: a cluster (1, 2, 4 or 8 CTAs) per segment, a batch per warp in turn. Also zeroes the
// workspace header (no separate launch for that).
__global__ void __launch_bounds__(kThreads, 4)
    topk_cluster_kernel(const float* __restrict__ scores, const int64_t* __restrict__ off, int k,
                        int32_t* __restrict__ out_i, float* __restrict__ out_s, unsigned char* __restrict__ header)
{
    __shared__ unsigned long long buf[kWarps][64], lists[kWarps][kMaxK];
    if (blockIdx.x == 0) header[threadIdx.x] = 0;
    cg::cluster_group cluster = cg::this_cluster();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int64_t s = blockIdx.x / ranks;
    const int64_t b = off[s];
    const Segment seg(scores + b, (int)(off[s + 1] - b));
    // warps that have a batch: the first ceil(n4 / 128) of the cluster's (and always the first)
    const int batches = (seg.n4 + kBatchF4 - 1) / kBatchF4;
    const int here = min(max(batches - rank * kWarps, 0), kWarps);
    const int used = max(1, min((batches + kWarps - 1) / kWarps, ranks));  // CTAs with one
    WarpList l(buf[warp], k, lane);
    if (warp < max(here, 1)) l.scan(seg, rank * kWarps + warp, ranks * kWarps, rank == 0 && warp == 0);
    if (here > 1) {
        if (lane < kMaxK) lists[warp][lane] = l.list;
        __syncthreads();
        if (warp == 0) l.list = merge_lists(lists, here, lane);
    }
    if (used > 1) {  // the same for all CTAs of the cluster
        __syncthreads();
        if (warp == 0 && lane < kMaxK) lists[0][lane] = l.list;
        cluster.sync();
        if (rank == 0 && warp == 0)
            for (int r = 1; r < used; ++r) {
                const unsigned long long* p = cluster.map_shared_rank(&lists[0][0], r);
                l.list = merge32(l.list, lane < kMaxK ? p[lane] : kNone, lane);
            }
        cluster.sync();  // a CTA's lists are read until here
    }
    if (rank == 0 && warp == 0) l.write(out_i + s * k, out_s + s * k);
}

// A warp per segment from as many segments as CTAs are resident on; below that a CTA per segment, and as
// many CTAs (2, 4, 8) as there is room for. 64 segments of 16,384 scores (8 CTAs each): 22.8 -> 8.8 us, of
// 262,144: 143 -> 17.5 us; 600 of 16,384 (1 CTA each) 24.2 -> 11.9 us, where a warp each takes 17; 1,200 of 64
// (a warp each): 6.8 -> 4.7 us, where a CTA each takes 10.
// With few more segments than CTAs resident, a CTA owns two or four of them instead of eight, so that all SMs have
// some (700 of 65,536, k = 5: 39 us on 350 CTAs, 97 on 88; of 16,384: 23 both).
int launch(const float* scores, const int64_t* off, int64_t n_seg, int k, int32_t* oi, float* os, void* workspace,
           cudaStream_t st)
{
    static std::atomic<int> per_sm_cache[tune::kMaxDevices];
    int per_sm = 0;
    int rc = tune::blocks_per_sm(per_sm_cache, reinterpret_cast<const void*>(topk_warp_kernel), kThreads, &per_sm);
    if (rc) return rc;
    const int sms = tune::device_sm_count();
    if (sms <= 0) return tune::fail(TUNE_ECUDA, "tune_topk: cannot query the SM count");
    const int64_t cap = (int64_t)sms * per_sm;
    if (n_seg > cap) {
        const int per_log = n_seg <= 2 * cap ? 1 : n_seg <= 4 * cap ? 2 : 3;
        const int64_t need = (n_seg + (1 << per_log) - 1) >> per_log;
        topk_warp_kernel<<<(int)(need < cap ? need : cap), kThreads, 0, st>>>(scores, off, n_seg, k, per_log, oi, os,
                                                                             static_cast<unsigned char*>(workspace));
        TUNE_CUDA_TRY(cudaGetLastError(), "tune_topk: kernel launch");
        return TUNE_OK;
    }
    int c = 1;
    while (c < 8 && n_seg * c * 2 <= cap) c *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_seg * c));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    TUNE_CUDA_TRY(cudaLaunchKernelEx(&cfg, topk_cluster_kernel, scores, off, k, oi, os, static_cast<unsigned char*>(workspace)),
                  "tune_topk: kernel launch");
    return TUNE_OK;
}

}  // namespace

extern "C" int tune_topk(const float* scores, const int64_t* seg_offsets, int64_t n_seg, int32_t k,
                         int32_t* topk_idx, float* topk_score, void* workspace, size_t ws_bytes,
                         tune_stream_t stream)
{
    tune::clear_error();
    if (k < 1 || k > 16) return tune::fail(TUNE_EINVAL, "k = %d outside [1, 16]", k);
    if (n_seg < 0) return tune::fail(TUNE_EINVAL, "n_seg < 0");
    if (!workspace) return tune::fail(TUNE_EINVAL, "workspace is NULL");
    if (ws_bytes < tune_workspace_bytes(TUNE_CALL_TOPK, n_seg, k))
        return tune::fail(TUNE_ENOMEM, "workspace too small");
    if (n_seg > 0 && (!scores || !seg_offsets || !topk_idx || !topk_score))
        return tune::fail(TUNE_EINVAL, "scores, seg_offsets and outputs must be non-NULL");
    if ((reinterpret_cast<uintptr_t>(scores) & 3) != 0)
        return tune::fail(TUNE_EINVAL, "scores must be 4-byte aligned");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (n_seg == 0) {
        TUNE_CUDA_TRY(cudaMemsetAsync(workspace, 0, tune::kWorkspaceHeader, s), "tune_topk: status reset");
        return TUNE_OK;
    }
    return launch(scores, seg_offsets, n_seg, k, topk_idx, topk_score, workspace, s);
}
