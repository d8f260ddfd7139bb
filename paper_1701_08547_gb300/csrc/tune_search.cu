// tune_search: random and Nelder-Mead simplex search over each kernel's tuning space,
// optionally restricted to a subset of its thread counts (the statically pruned space),
// with the analytic cost as the objective. The paper's autotuner explores the space
// left after static pruning with one of its search methods, exhaustive, random or
// Nelder-Mead simplex (Sections III-C and IV-C); here the objective is the static model itself,
// so a search costs no runs of the kernel.
//
// One thread per kernel descriptor: a search is a sequential chain of evaluations.
// A point is a rank vector (a0, a1, a2, a3) over the searched lists of thread counts,
// grid sizes, unroll factors and carveouts; its objective is the FP32 cost of
// point_cost() (+inf without a valid configuration) and points are ordered by
// (cost, canonical index), the canonical index being the point's index in the
// kernel's full space (as in tune_eval).
//
// What bounds it is the chain: some 55 evaluations one after the other, 128 at most. So an
// evaluation is a handful of lookups: the architecture's tables (eval_tables.cuh) in
// shared memory, and per thread the kernel's cost sums and register limits by unroll
// rank, its G_S by carveout rank (a register) and its axis positions by rank. And the
// Nelder-Mead steps are a state machine with one evaluation per turn, at one place for
// all lanes, the simplex in shared memory and its five (cost, index) keys in registers.
// (Pricing each point from scratch, some 400 instructions at five places where the lanes of
// a warp arrived at different times, took 1,270 us for 100,000 pruned dense kernels with a
// budget of 128 evaluations; now 254, some 400 instructions of state handling per turn being
// what is left.)
//
// Random search: evaluation j draws a_d = below(draw(4 j + d), n_d).
// Nelder-Mead: vertices are fixed-point rank vectors (8 fractional bits) rounded to
// the nearest rank and clamped to the list; reflection 1, expansion 2, contraction
// 1/2 (outside or inside), shrink 1/2 towards the best vertex, all in integer
// arithmetic with floor shifts; the search stops when the evaluation budget is spent
// or a shrink leaves every vertex on one point. Both report the best point seen.
#include <stdint.h>

#include "eval_tables.cuh"
#include "tune_internal.h"

using namespace tune_dev;

namespace {

constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
constexpr int kThreadsS = 128;
constexpr int kQ = 8;  // fractional bits of the simplex coordinates

// SplitMix64 finaliser (Steele, Lea and Flood, 2014).
__device__ __forceinline__ uint64_t mix64(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Draw j of kernel i, mapped to [0, n): SplitMix64 output of the state
// mix64(seed) + (i 2^32 + j + 1) gamma, top 32 bits times n, shifted down 32.
__device__ __forceinline__ int draw_below(uint64_t key, int64_t i, uint32_t j, int n)
{
    const uint64_t x = mix64(key + ((uint64_t)i * 4294967296ull + (uint64_t)j + 1ull) * kGamma);
    return (int)(((x >> 32) * (uint64_t)n) >> 32);
}

// (cost, canonical index) keys: costs are >= 0 (or +inf), so their bit patterns order like the values.
__device__ __forceinline__ uint64_t make_key(float c, int idx) { return ((uint64_t)__float_as_uint(c) << 32) | (uint32_t)idx; }
constexpr uint64_t kNoPoint = 0x7f80000000000000ull;  // +inf, index 0: no point without a configuration is below it

// What a thread keeps in shared memory (element [i] of every thread side by side).
struct ThreadTables {
    float cnm[8][kThreadsS];         // C_nm by unroll rank
    uint32_t regs[8][kThreadsS];     // register-limited warps | largest W_B that fits << 7 | R << 15, by unroll rank
    int v[5][4][kThreadsS];          // simplex vertices, fixed point
    unsigned char tpos[32][kThreadsS], gpos[16][kThreadsS];  // axis positions by rank
};

struct SearchParams {
    tune_arch a;
    tune_axes x;
    CtaTables tab;
};

struct Searcher {
    const tune_arch& a;
    const CtaTables& ct;
    ThreadTables& t;
    const int tid;
    uint32_t tm;     // the kernel's full thread-count mask (canonical index)
    int n[4];        // lengths of the searched lists
    int nG, nU, nC;  // full axis counts of the kernel's space
    float cm;        // C_m (the unroll factor does not enter it)
    uint32_t gs;     // G_S by carveout rank, a byte each
    bool simple;     // per-warp register allocation, R > 0 for every unroll factor
    uint64_t best = kNoPoint;
    int evals = 0;

    // Key of a rank vector; records the best point seen.
    __device__ __forceinline__ uint64_t eval(const int (&r)[4])
    {
        const int tp = t.tpos[r[0]][tid], gp = t.gpos[r[1]][tid], wb = ct.wb[tp];
        const uint32_t ru = t.regs[r[2]][tid];
        const int warps = (int)(ru & 0x7fu), wbmax = (int)((ru >> 7) & 0xffu);
        const int gr = simple ? (wb > wbmax ? 0 : (int)ct.divt[warps][tp])
                              : reg_blocks(a, ct, (int)(ru >> 15), wb, tp, warps, wbmax);
        const int B = min(min(ct.gw[tp], gr), (int)((gs >> (8 * r[3])) & 0xffu));
        const float X = __fmul_rn(__fmaf_rn(cm, ct.hide[B * wb], t.cnm[r[2]][tid]), ct.lane[tp]);
        float c = __fmul_rn(X, ct.ipar[max(B, 1) - 1][gp]);
        if (B <= 0 || !(c == c)) c = __int_as_float(0x7f800000);  // NaN ranks as +inf
        const int t_full = __popc(tm & ((1u << tp) - 1u));
        const uint64_t key = make_key(c, ((t_full * nG + r[1]) * nU + r[2]) * nC + r[3]);
        ++evals;
        best = min(best, key);
        return key;
    }

    __device__ void random(uint64_t key, int64_t kid, int budget)
    {
        for (int j = 0; j < budget; ++j) {
            int r[4];
#pragma unroll
            for (int d = 0; d < 4; ++d) r[d] = draw_below(key, kid, (uint32_t)(4 * j + d), n[d]);
            eval(r);
        }
    }

    // Fixed-point coordinate d -> nearest rank, clamped to the list.
    __device__ __forceinline__ int rank_of(int v, int d) const
    {
        return min(max((v + (1 << (kQ - 1))) >> kQ, 0), n[d] - 1);
    }

    __device__ void nelder_mead(uint64_t key, int64_t kid, int budget)
    {
        enum { kInit, kReflect, kExpand, kContract, kShrink };
        // initial simplex: x0 and one step of max(1, n_d / 4) ranks along each axis
        // (backwards where forwards leaves the list)
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const int x0 = draw_below(key, kid, (uint32_t)d, n[d]) << kQ;
            const int s = max(1, n[d] >> 2) << kQ;
#pragma unroll
            for (int j = 0; j < 5; ++j) t.v[j][d][tid] = x0;
            t.v[d + 1][d][tid] = x0 + s <= ((n[d] - 1) << kQ) ? x0 + s : x0 - s;
        }
        uint64_t K[5], kr = 0, ksw = 0;  // the vertices' keys; the one to beat or to store; the second worst's
        int sum[4], vw[4], c[4], x[4];   // sum of the vertices, worst vertex, centroid of the others, point to evaluate
        int state = kInit, j = 0, b = 0, w = 0;  // j: vertex being evaluated (kInit, kShrink); best, worst
#pragma unroll
        for (int i = 0; i < 5; ++i) K[i] = 0;
#pragma unroll
        for (int d = 0; d < 4; ++d) x[d] = t.v[0][d][tid], sum[d] = vw[d] = c[d] = 0;
        while (evals < budget) {
            int r[4];
#pragma unroll
            for (int d = 0; d < 4; ++d) r[d] = rank_of(x[d], d);
            const uint64_t kx = eval(r);
            bool next = false;  // the next step starts, after
            int put = -1;       // x, of key kr, has taken the place of this vertex
            if (state == kReflect) {
                kr = kx;
                uint64_t kb = K[0], kw = K[0];
#pragma unroll
                for (int i = 1; i < 5; ++i) {
                    kb = b == i ? K[i] : kb;
                    kw = w == i ? K[i] : kw;
                }
                if (kx < kb) {
                    // (with the budget spent, the simplex is not looked at again)
                    state = kExpand;
#pragma unroll
                    for (int d = 0; d < 4; ++d) x[d] = 3 * c[d] - 2 * vw[d];
                } else if (kx < ksw) {
                    put = w;
                } else {
                    // contraction, outside if the reflection beats the worst, else inside: has to beat kr
                    const bool outside = kx < kw;
                    state = kContract;
                    kr = outside ? kx : kw;
#pragma unroll
                    for (int d = 0; d < 4; ++d) x[d] = c[d] + (((outside ? x[d] : vw[d]) - c[d]) >> 1);
                }
            } else if (state == kExpand) {
                const bool better = kx < kr;  // else the reflection, 2 c - w
                kr = better ? kx : kr;
#pragma unroll
                for (int d = 0; d < 4; ++d) x[d] = better ? x[d] : 2 * c[d] - vw[d];
                put = w;
            } else if (state == kContract) {
                if (kx < kr) {
                    kr = kx;
                    put = w;
                } else {
                    state = kShrink;
                    j = -1;
                }
            } else {
                kr = kx;
                put = j;
            }
            if (put >= 0) {
                next = true;
#pragma unroll
                for (int i = 0; i < 5; ++i) K[i] = put == i ? kr : K[i];
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    sum[d] += x[d] - vw[d];
                    t.v[put][d][tid] = x[d];
                }
            }
            if (state == kInit) {  // (vw is 0: the vertices add up)
                next = ++j == 5;
                if (!next)
#pragma unroll
                    for (int d = 0; d < 4; ++d) x[d] = t.v[j][d][tid];
            } else if (state == kShrink) {  // the next vertex moves halfway to the best
                next = false;
                if (++j == b) ++j;
                if (j < 5) {
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        const int vb = t.v[b][d][tid];
                        vw[d] = t.v[j][d][tid];
                        x[d] = vb + ((vw[d] - vb) >> 1);
                    }
                } else {
                    bool same = true;
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        const int rb = rank_of(t.v[b][d][tid], d);
#pragma unroll
                        for (int i = 0; i < 5; ++i) same = same && rank_of(t.v[i][d][tid], d) == rb;
                    }
                    if (same) return;
                    next = true;
                }
            }
            if (next) {
                // best, worst and second worst by (cost, index, vertex number); the reflection
                b = w = 0;
                uint64_t kb = K[0], kw = K[0];
                ksw = 0;
#pragma unroll
                for (int i = 1; i < 5; ++i) {
                    if (K[i] < kb) b = i, kb = K[i];
                    const bool worst = K[i] >= kw;
                    ksw = worst ? kw : (K[i] > ksw ? K[i] : ksw);
                    if (worst) w = i, kw = K[i];
                }
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    vw[d] = t.v[w][d][tid];
                    c[d] = (sum[d] - vw[d]) >> 2;
                    x[d] = 2 * c[d] - vw[d];
                }
                state = kReflect;
            }
        }
    }
};

// Seven CTAs per SM: 152 x 7 x 128 threads hold 100,000 kernels at once.
__global__ void __launch_bounds__(kThreadsS, 7)
    tune_search_kernel(const __grid_constant__ SearchParams p, const int4* __restrict__ descs, int64_t n_kernels,
                       int method, int budget, uint64_t key, const uint32_t* __restrict__ t_keep,
                       int32_t* __restrict__ best_idx, float* __restrict__ best_cost, int32_t* __restrict__ evals,
                       int* __restrict__ status)
{
    __shared__ CtaTables ct;
    __shared__ ThreadTables tt;
    copy_cta_tables(p.tab, ct);
    __syncthreads();
    const int tid = threadIdx.x;
    const int64_t kid = (int64_t)blockIdx.x * kThreadsS + tid;
    if (kid >= n_kernels) return;
    int4 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = __ldg(descs + kid * 4 + q);
    Desc kd;
    unpack(v, kd);
    const uint32_t mt = kd.tm & (t_keep ? t_keep[kid] : 0xffffffffu);
    Searcher s{p.a, ct, tt, tid, kd.tm, {__popc(mt), __popc(kd.gm), __popc(kd.um), __popc(kd.cm)}};
    s.nG = s.n[1];
    s.nU = s.n[2];
    s.nC = s.n[3];
    const bool bad = desc_bad(kd, p.x);
    if (bad) atomicOr(status, tune::kStatusInvalid);
    if (!bad && s.n[0] > 0 && s.n[1] > 0 && s.n[2] > 0 && s.n[3] > 0) {
        // the kernel's tables
        int r = 0;
        for (uint32_t m = mt; m; m &= m - 1u) tt.tpos[r++][tid] = (unsigned char)(__ffs(m) - 1);
        r = 0;
        for (uint32_t m = kd.gm; m; m &= m - 1u) tt.gpos[r++][tid] = (unsigned char)(__ffs(m) - 1);
        r = 0;
        for (uint32_t m = kd.um; m; m &= m - 1u, ++r) {
            const int U = p.x.u[__ffs(m) - 1], R = kd.r0 + 4 * (U - 1);
            float cnm;
            unit_costs(kd.n, kd.d, U, ct.rcp, p.a.work_scale, cnm, s.cm);
            int warps, wbmax;
            if (R >= 0 && R < 256) {
                warps = ct.rwarps[R];
                wbmax = ct.rwbmax[R];
            } else {
                reg_params(p.a, R, warps, wbmax);
            }
            tt.cnm[r][tid] = cnm;
            // W_B is at most 128 (T <= 4,096) and R above 2^17 - 1 is above every limit of registers per thread
            tt.regs[r][tid] = (uint32_t)warps | ((uint32_t)min(wbmax, 255) << 7) | ((uint32_t)min(R, (1 << 17) - 1) << 15);
        }
        s.gs = 0;
        r = 0;
        for (uint32_t m = kd.cm; m; m &= m - 1u, ++r)
            s.gs |= (uint32_t)min(smem_blocks_from(p.a, ct, kd.s0, __ffs(m) - 1), 255) << (8 * r);
        s.simple = p.a.reg_alloc_mode == 0 && kd.r0 > 0;
        if (method == TUNE_SEARCH_RANDOM)
            s.random(key, kid, budget);
        else
            s.nelder_mead(key, kid, budget);
    }
    const float cost = __uint_as_float((uint32_t)(s.best >> 32));
    best_idx[kid] = s.best < kNoPoint ? (int)(uint32_t)s.best : -1;
    best_cost[kid] = cost;
    evals[kid] = s.evals;
}

}  // namespace

extern "C" int tune_search(const tune_arch* arch, const tune_axes* axes, const tune_kernel_desc* descs,
                           int64_t n_kernels, int32_t method, int32_t budget, uint64_t seed, const uint32_t* t_keep,
                           int32_t* best_idx, float* best_cost, int32_t* evals, void* workspace, size_t ws_bytes,
                           tune_stream_t stream)
{
    tune::clear_error();
    if (!arch || !axes) return tune::fail(TUNE_EINVAL, "arch and axes must be non-NULL host pointers");
    if (method != TUNE_SEARCH_RANDOM && method != TUNE_SEARCH_NELDER_MEAD)
        return tune::fail(TUNE_EINVAL, "method %d is neither TUNE_SEARCH_RANDOM nor TUNE_SEARCH_NELDER_MEAD", method);
    if (budget < 1 || budget > (1 << 20)) return tune::fail(TUNE_EINVAL, "budget %d outside [1, 2^20]", budget);
    if (n_kernels < 0) return tune::fail(TUNE_EINVAL, "n_kernels < 0");
    if (!workspace || ws_bytes < (size_t)tune::kWorkspaceHeader)
        return tune::fail(TUNE_ENOMEM, "workspace smaller than %d bytes", tune::kWorkspaceHeader);
    if (n_kernels > 0 && (!descs || !best_idx || !best_cost || !evals))
        return tune::fail(TUNE_EINVAL, "descs and outputs must be non-NULL");
    if ((reinterpret_cast<uintptr_t>(descs) & 15) != 0) return tune::fail(TUNE_EINVAL, "descs must be 16-byte aligned");
    int rc = tune::validate_inputs(arch, axes);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    TUNE_CUDA_TRY(cudaMemsetAsync(workspace, 0, tune::kWorkspaceHeader, s), "tune_search: status reset");
    if (n_kernels == 0) return TUNE_OK;
    // key = mix64(seed), computed on the host with the same finaliser
    uint64_t z = seed;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    const uint64_t key = z ^ (z >> 31);
    const int64_t blocks = (n_kernels + kThreadsS - 1) / kThreadsS;
    SearchParams p;
    p.a = *arch;
    p.x = *axes;
    tune::eval_tables(p.a, p.x, p.tab);
    tune_search_kernel<<<(unsigned)blocks, kThreadsS, 0, s>>>(p, reinterpret_cast<const int4*>(descs), n_kernels, method,
                                                              budget, key, t_keep, best_idx, best_cost, evals,
                                                              static_cast<int*>(workspace));
    TUNE_CUDA_TRY(cudaGetLastError(), "tune_search: kernel launch");
    return TUNE_OK;
}
