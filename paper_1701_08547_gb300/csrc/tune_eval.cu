// tune_eval: occupancy (Eqs. 1-5) + instruction-mix cost (Eq. 6 with launch-shape
// terms) over every point of every kernel's tuning space, then per-kernel top-k.
//
// Work decomposition (GB300, CUDA cores only; the path is integer/FP32 issue-bound):
//  * one warp evaluates one kernel descriptor; the warps of a CTA (eight) take its
//    descriptors from a counter (grid = SMs x resident CTAs), or a queue hands them
//    out over the whole grid;
//  * per CTA, once: a copy of the tables that depend only on the architecture row and
//    the axes (W_B, G_W, lane by thread count; hide by W*; waves/slots factor by
//    (B*, G); floor(w / W_B) for the register limit), which the host builds;
//  * per kernel, lane-parallel: the per-unroll cost sums C_nm(U), C_m(U)
//    (compensated FP32 sums), register-limited warps, per-carveout G_S, and
//    the (T, U) block limit min(G_W, G_R);
//  * pre-pass: a lane walks (T, U, C) triples; occupancy B*, W* come from
//    two table lookups and a min (grid size does not enter Eqs. 1-5); every
//    grid size G of a triple costs X(T,U,C) * ipar(B*, G), and since a product
//    by X > 0 is monotone under round-to-nearest the triple's cheapest point
//    is exactly X * min_G ipar(B*, G): one FP32 multiply per triple. A value
//    that k distinct triple minima do not exceed (tau0, from each lane's two
//    smallest (T, U)-pair minima counted with their multiplicities) bounds the
//    kernel's k-th best cost; each triple's minimum is kept in shared memory;
//  * main pass: lanes scan the minima; only triples that can still beat the
//    bound are re-evaluated, and the warp merges their grid sizes in
//    increasing (cost, index) order into a warp-wide exact top-k list (lane j
//    holds the j-th best); ties go to the lower canonical index.
//  * with TUNE_EMIT_POINTS every point's B*, W* and cost is written after that, in
//    canonical order.
//
// Bound by issue slots (about 80 % used). 100,000 dense kernels, k = 10: 216 -> 196 us; 1,000,000
// uneven ones, k = 5: 1,434 -> 1,238 us; 317,078 of 128 points, k = 15: 1,267 -> 672 us, from walks over
// the kernel's grid sizes by a mask of places instead of a scan of the row (1,361 us uneven), the
// list of a batch left in shared memory until it is complete, candidates kept in triple order (so that
// equal costs come in lane order and leave together), equal bounds counted together, two carveouts per
// packed FP32 operation, and the descriptor and the unroll tables read as 16-byte words.
#include <math.h>
#include <stdint.h>

#include <string.h>

#include <algorithm>
#include <condition_variable>
#include <limits>
#include <mutex>

#include "eval_tables.cuh"
#include "f32x2.cuh"
#include "pdl.cuh"
#include "tune_internal.h"

namespace {

using namespace tune_dev;
using f32x2::fma2;
using f32x2::mul2;

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr unsigned kFull = 0xffffffffu;

constexpr int kMaxArch = 8;  // architecture rows of one tune_eval_archs call

// Parameters of one launch. The CTA tables depend on the architecture row and the axes only, so the host
// builds them and passes them here, 6.6 KB of kernel parameters each CTA copies to shared memory.
struct EvalParams {
    tune_arch a;
    tune_axes x;
    int64_t n_kernels;
    int k;
    int chunk;        // dynamic work queue: kernels per grab (0 = each CTA its own descriptors)
    int group;        // emitting: descriptors a CTA takes at a time (1..8)
    int next_row;     // another row of the same sweep is launched next
    CtaTables tab;
};

// (T, U, C) triples whose points the emitting pass writes at a time: what the ranking's keys leave room for.
constexpr int kEmitTriples = 240;
// Points of a space that the warp which ranked it writes by itself; those of larger ones are shared by the CTA
// (200,000 kernels of 128 points each: 511 us by themselves, 824 shared).
constexpr int kEmitAlone = 2048;

struct WarpTables {
    alignas(8) float iparmin[kMaxB + 1];  // by B*: min over the kernel's grid sizes of ipar(B*, G); [0] = NaN
    unsigned short places[kMaxB + 1];  // by B*: the kernel's grid sizes as places in rperm (not for a full set)
    unsigned char gwr[32][8];  // min(G_W, G_R) by (t rank, u rank)
    // by u rank: C_nm; C_m; register-limited warps | (largest W_B that fits) << 8; R (the last two as bits)
    float4 uinfo[8];
    int gs[4];               // G_S by c rank
    int4 tinfo[32];          // by t rank: W_B, lane efficiency (float bits), t position, G_W
    int gpos[16];            // g position by g rank
    // emitting pass: the space's axis sizes (nT = 0: nothing to write), whether the (T, U) block limit is
    // formed in place, and the first point's place in the arrays
    int nT, nG, nU, nC, simple;
    int64_t off;
    union {
        int4 desc[4];        // the descriptor's words, before the ranking pass
        float key[32 * 32];  // ranking pass: each triple's minimum cost, by (row, lane)
        struct {             // emitting pass, after the ranking:
            float iparc[kMaxB][kIparStride];  // ipar rows compacted to the kernel's grid sizes
            // of the triples whose points are being written: X (+inf where B* = 0), and B* | W* << 8 |
            // word offset of the ipar row << 16
            float2 tri[kEmitTriples];
        };
    };
};

// (cost, index) keys ordered lexicographically; costs are >= 0, so their bit
// patterns order like the values.
__device__ __forceinline__ bool key_less(float c, int i, float c2, int i2)
{
    return c < c2 || (c == c2 && i < i2);
}

template <int N>
struct IntC {
    static constexpr int value = N;
};

// floor(n / d) for 0 <= n < 8192 and 1 <= d <= 32, given rcp = 1/d rounded to
// nearest: (n + 1/2) / d lies at least 1/64 away from an integer, far more than
// the rounding error of the product, so truncation is exact.
__device__ __forceinline__ int small_div(int n, float rcp)
{
    return __float2int_rz(__fmul_rn((float)n + 0.5f, rcp));
}

// Warp-wide top-k list: lane j < k holds the j-th best (cost, index), ascending.
// Inserts one key (the same on every lane); returns nothing, updates the list
// and the k-th key (tau) on every lane.
__device__ __forceinline__ void warp_list_insert(float& lc, int& li, float& tau_c, int& tau_i, float c,
                                                 int i, int k, int lane)
{
    const unsigned below = __ballot_sync(kFull, lane < k && key_less(lc, li, c, i));
    const int pos = __popc(below);
    const float up_c = __shfl_up_sync(kFull, lc, 1);
    const int up_i = __shfl_up_sync(kFull, li, 1);
    if (lane < k) {
        if (lane == pos) {
            lc = c;
            li = i;
        } else if (lane > pos) {
            lc = up_c;
            li = up_i;
        }
    }
    tau_c = __shfl_sync(kFull, lc, k - 1);
    tau_i = __shfl_sync(kFull, li, k - 1);
}

// min(G_W, G_R) of (t rank, u rank); ti = tinfo[t rank], ui = uinfo[u rank].
__device__ __forceinline__ int block_limit_of(const CtaTables& ct, const WarpTables& w, bool simple, int t_r, const int4& ti,
                                              int u_r, const float4& ui)
{
    if (!simple) return w.gwr[t_r][u_r];
    const int ru = __float_as_int(ui.z);
    return min(ti.w, ti.x > (ru >> 8) ? 0 : (int)ct.divt[ru & 0xff][ti.z]);
}

// Writes B*, W* and cost of the points of thread-count ranks t_beg .. t_end - 1 of the kernel whose tables are w,
// in canonical order (G between T and the (U, C) pairs), so that the warp's stores are whole lines whatever the
// kernel's axes; tris: kEmitTriples entries of the warp's own.
__device__ __forceinline__ void emit_points(const CtaTables& ct, const WarpTables& w, float2* tris, int t_beg, int t_end,
                                            int lane, int32_t* __restrict__ pt_b, int32_t* __restrict__ pt_w,
                                            float* __restrict__ pt_c)
{
    if (t_beg >= t_end) return;  // (also where there is no kernel: the other fields are not set then)
    const float kInf = __int_as_float(0x7f800000);
    const int nG = w.nG, nC = w.nC, nUC = w.nU * nC, g_stride = nG * nUC;
    const bool simple = w.simple != 0;
    if (nUC >= 8 && (nUC & (nUC - 1)) == 0) {
        // 8, 16 or 32 (U, C) pairs: a lane keeps its triple and walks the grid sizes, 32 / nUC of them per step
        // of 32 consecutive points (a third of the instructions of the general walk)
        const int uc_r = lane & (nUC - 1), g0 = lane / nUC, dg = 32 / nUC;
        const int u_r = uc_r / nC, c = uc_r - u_r * nC;
        const float4 ui = w.uinfo[u_r];
        const float cnm = ui.x, cmv = ui.y;
        const int gs = w.gs[c];
        int64_t at = w.off + (int64_t)t_beg * g_stride + lane;
        for (int t_r = t_beg; t_r < t_end; ++t_r, at += g_stride) {
            const int4 ti = w.tinfo[t_r];
            const int B = min(block_limit_of(ct, w, simple, t_r, ti, u_r, ui), gs), W = B * ti.x;
            const float X = B > 0 ? __fmul_rn(__fmaf_rn(cmv, ct.hide[W], cnm), __int_as_float(ti.y)) : kInf;
            const float* row = w.iparc[max(B, 1) - 1];
            int64_t q = at;
#pragma unroll 4
            for (int g = g0; g < nG; g += dg, q += 32) {
                if (pt_b) __stcs(pt_b + q, B);
                if (pt_w) __stcs(pt_w + q, W);
                if (pt_c) __stcs(pt_c + q, __fmul_rn(X, row[g]));
            }
        }
        return;
    }
    // a stretch of thread counts at a time whose triples are formed first; a lane writes four consecutive points
    // with 16-byte stores where the arrays' alignment allows it
    const float rcp_c = ct.rcpn[nC], rcp_uc = ct.rcpn[nUC], rcp_g = ct.rcpn[nG];
    const int t_step = kEmitTriples / nUC;
    const int64_t off = w.off;
    // points (of 4 bytes) to the next 16-byte boundary, per array; one where they agree
    const auto lead = [&](const void* q) {
        return q ? (int)((4u - (unsigned)(reinterpret_cast<uintptr_t>(q) >> 2) - (unsigned)off) & 3u) : -1;
    };
    const int lb = lead(pt_b), lw = lead(pt_w), lc = lead(pt_c), lany = max(lb, max(lw, lc));
    const bool vec = (lb < 0 || lb == lany) && (lw < 0 || lw == lany) && (lc < 0 || lc == lany);
    for (int t0 = t_beg; t0 < t_end; t0 += t_step) {
        const int n_tri = min(t_step, t_end - t0) * nUC;
        for (int tri = lane; tri < n_tri; tri += 32) {
            const int t_r = small_div(tri, rcp_uc), uc_r = tri - t_r * nUC;
            const int u_r = small_div(uc_r, rcp_c), c = uc_r - u_r * nC;
            const int4 ti = w.tinfo[t0 + t_r];
            const float4 ui = w.uinfo[u_r];
            const int B = min(block_limit_of(ct, w, simple, t0 + t_r, ti, u_r, ui), w.gs[c]), W = B * ti.x;
            const float X = __fmul_rn(__fmaf_rn(ui.y, ct.hide[W], ui.x), __int_as_float(ti.y));
            tris[tri] = make_float2(B > 0 ? X : kInf, __int_as_float(B | (W << 8) | (((max(B, 1) - 1) * kIparStride) << 16)));
        }
        __syncwarp();
        const int n_pt = n_tri * nG;  // at most 3,840
        const int64_t at0 = off + (int64_t)t0 * g_stride;
        // walks the points p, p + 1, ... of the stretch
        int uc_r = 0, g_r = 0, tri = 0;
        auto seek = [&](int p) {
            const int q = small_div(p, rcp_uc), t_r = small_div(q, rcp_g);
            uc_r = p - q * nUC;
            g_r = q - t_r * nG;
            tri = t_r * nUC + uc_r;
        };
        auto point = [&](int& B, int& W, float& c) {
            const float2 t = tris[tri];
            const unsigned bw = __float_as_uint(t.y);
            B = (int)(bw & 0xffu);
            W = (int)((bw >> 8) & 0xffu);
            c = __fmul_rn(t.x, (&w.iparc[0][0])[(bw >> 16) + g_r]);
            ++tri;
            if (++uc_r == nUC) {
                uc_r = 0;
                if (++g_r == nG)
                    g_r = 0;
                else
                    tri -= nUC;
            }
        };
        auto write1 = [&](int p) {
            int B, W;
            float c;
            seek(p);
            point(B, W, c);
            if (pt_b) pt_b[at0 + p] = B;
            if (pt_w) pt_w[at0 + p] = W;
            if (pt_c) pt_c[at0 + p] = c;
        };
        if (vec) {
            const int head = min((lany - t0 * g_stride) & 3, n_pt), n4 = (n_pt - head) >> 2;
            const int p1 = lane < head ? lane : 4 * n4 + lane;  // at most 3 + 3 single points, before and after
            if (lane < head + 3 && p1 < n_pt) write1(p1);
            for (int f = lane; f < n4; f += 32) {
                const int p = head + 4 * f;
                int4 B, W;
                float4 c;
                seek(p);
                point(B.x, W.x, c.x);
                point(B.y, W.y, c.y);
                point(B.z, W.z, c.z);
                point(B.w, W.w, c.w);
                if (pt_b) __stcs(reinterpret_cast<int4*>(pt_b + at0 + p), B);
                if (pt_w) __stcs(reinterpret_cast<int4*>(pt_w + at0 + p), W);
                if (pt_c) __stcs(reinterpret_cast<float4*>(pt_c + at0 + p), c);
            }
        } else {
            for (int p = lane; p < n_pt; p += 32) write1(p);
        }
        __syncwarp();
    }
}

template <bool EMIT>
__global__ void __maxnreg__(64)
    tune_eval_kernel(const __grid_constant__ EvalParams p, const int4* __restrict__ descs,
                     int32_t* __restrict__ topk_idx, float* __restrict__ topk_cost,
                     int32_t* __restrict__ pt_b, int32_t* __restrict__ pt_w,
                     float* __restrict__ pt_c, const int64_t* __restrict__ pt_off,
                     int* __restrict__ status, unsigned long long* __restrict__ queue)
{
    __shared__ CtaTables ct;
    __shared__ WarpTables wts[kWarps];
    __shared__ int taken;
    const tune_arch& a = p.a;
    // a row of tune_eval_archs before the last: the next row's CTAs may take the places that this one's leave
    // (independent launches, pdl.cuh)
    if (p.next_row) pdl::grid_dep_launch();
    copy_cta_tables(p.tab, ct);
    if (threadIdx.x == 0) taken = kWarps;
    __syncthreads();

    const tune_axes& x = p.x;
    const int lane = threadIdx.x & 31;
    WarpTables& w = wts[threadIdx.x >> 5];
    const float kInf = __int_as_float(0x7f800000);
    const int k = p.k;
    const int64_t n_k = p.n_kernels;
    const uint32_t g_ok = (1u << x.n_g) - 1u;

    // Work distribution: each CTA owns 8 consecutive descriptors of every 8 x grid, which its warps take one after the
    // other from a counter in shared memory (a warp with large spaces takes fewer); or (chunk > 0) a queue of the whole
    // grid from which each warp takes `chunk` consecutive descriptors at a time. The next descriptor's words, and the
    // number of the one (in queue mode the start of the chunk) after it, are fetched while the current descriptor is
    // evaluated.
    const int64_t stride = (int64_t)gridDim.x * kWarps;
    unsigned long long grabbed = 0;  // lane 0: start of the next chunk, or number of the CTA's descriptor
    auto grab = [&]() {
        if (lane == 0) grabbed = p.chunk ? atomicAdd(queue, (unsigned long long)p.chunk) : (unsigned)atomicAdd(&taken, 1);
    };
    auto grabbed_kid = [&]() {
        const unsigned long long i = __shfl_sync(kFull, grabbed, 0);
        return p.chunk ? (int64_t)i : (int64_t)(i / kWarps) * stride + (int64_t)blockIdx.x * kWarps + (int)(i % kWarps);
    };
    // ranks descriptor kid, whose four 16-byte words lanes 0..3 (mod 4) hold in v, on this warp
    auto rank = [&](const int64_t kid, const int4 v) {
        if (lane < 4) w.desc[lane] = v;
        __syncwarp();
        const int4 vw[4] = {w.desc[0], w.desc[1], w.desc[2], w.desc[3]};
        Desc kd;
        unpack(vw, kd);
        const int r0 = kd.r0, s0 = kd.s0;
        const uint32_t tm = kd.tm, gm = kd.gm, um = kd.um, cm = kd.cm;
        // (a count per lane: its words 0..6)
        const bool bad = __any_sync(kFull, (lane < 7 && count_bad(reinterpret_cast<const float*>(w.desc)[lane])) ||
                                               desc_fields_bad(kd, x));
        const int nT = __popc(tm), nG = __popc(gm), nU = __popc(um), nC = __popc(cm);
        if (bad || nT * nG * nU * nC == 0) {
            if (bad && lane == 0) atomicOr(status, tune::kStatusInvalid);
            if (lane < k) {
                topk_idx[kid * k + lane] = -1;
                topk_cost[kid * k + lane] = kInf;
            }
            __syncwarp();  // the descriptor's words are rewritten
            return;
        }
        const int nUC = nU * nC;
        const int g_stride = nG * nUC;

        // ---- per-axis tables, lane = axis position: per unroll the cost sums and
        // register limits, per carveout G_S.
        const uint32_t below = (1u << lane) - 1u;
        if (lane < 16 && ((gm >> lane) & 1u)) w.gpos[__popc(gm & below)] = lane;
        if (lane < 8 && ((um >> lane) & 1u)) {
            const int ur = __popc(um & below);
            const int U = x.u[lane];
            const int R = r0 + 4 * (U - 1);
            float cnm, cm_u;
            unit_costs(kd.n, kd.d, U, ct.rcp, a.work_scale, cnm, cm_u);
            int warps, wbmax;
            if (R >= 0 && R < 256) {
                warps = ct.rwarps[R];
                wbmax = ct.rwbmax[R];
            } else {
                reg_params(a, R, warps, wbmax);
            }
            w.uinfo[ur] = make_float4(cnm, cm_u, __int_as_float(warps | (wbmax << 8)), __int_as_float(R));
        }
        if (lane < 4 && ((cm >> lane) & 1u)) w.gs[__popc(cm & below)] = smem_blocks_from(a, ct, s0, lane);
        // Per-warp register allocation with R > 0 for every unroll (r0 > 0): the (T, U)
        // block limit is min(G_W, W_B > wbmax ? 0 : floor(warps / W_B)) and is formed
        // where it is used; otherwise (per-block allocation, R = 0) it is tabulated.
        const bool simple = a.reg_alloc_mode == 0 && r0 > 0;
        __syncwarp();
        // ---- per thread count (lane = t position): W_B, lane efficiency, G_W by t rank
        // (and the tabulated block limit min(G_W, G_R)).
        if ((tm >> lane) & 1u) {
            const int tr = __popc(tm & below);
            const int wb = ct.wb[lane];
            const int gw = ct.gw[lane];
            w.tinfo[tr] = make_int4(wb, __float_as_int(ct.lane[lane]), lane, gw);
            if (!simple) {
                for (int ur = 0; ur < nU; ++ur) {
                    const float4 ui = w.uinfo[ur];
                    const int ru = __float_as_int(ui.z);
                    const int gr = reg_blocks(a, ct, __float_as_int(ui.w), wb, lane, ru & 0xff, ru >> 8);
                    w.gwr[tr][ur] = (unsigned char)min(gw, gr);
                }
            }
        }
        auto block_limit = [&](int t_r, const int4& ti, int u_r, const float4& ui) {
            return block_limit_of(ct, w, simple, t_r, ti, u_r, ui);
        };
        // ---- by B* (lane = B* - 1): this kernel's grid sizes as places in the row's increasing order, and the
        // row's minimum over them, the first place's.
        const bool g_dense = gm == g_ok;
        const unsigned all_places = 0x10000u - (0x10000u >> x.n_g);
        if (lane == 0) w.iparmin[0] = __int_as_float(0x7fc00000);  // B* = 0: no valid configuration
        if (lane < kMaxB) {
            if (g_dense) {
                w.iparmin[lane + 1] = ct.iparmin[lane];
            } else {
                // (a warp-uniform trip count)
                unsigned pl = 0;
                const unsigned long long of = ct.place[lane];
                for (int j = 0; j < nG; ++j) pl |= 1u << ((unsigned)(of >> (4 * w.gpos[j])) & 15u);
                w.places[lane + 1] = (unsigned short)pl;
                w.iparmin[lane + 1] = ct.ipar[lane][ct.rperm[lane][31 - __clz(pl)]];
            }
        }
        __syncwarp();

        float lc = kInf;  // this lane's entry of the warp's top-k list (lanes < k)
        int li = -1;
        float tau_c = kInf;  // the list's k-th key
        int tau_i = -1;
        float tau0 = kInf;   // bound from the pre-pass

        // A lane's walk over the grid sizes of its candidate triple in increasing cost (the order of
        // X * ipar(B*, G) over G depends on B* only): the highest set bit of `places` is the next one. Points
        // are numbered t rank << 9 | g position << 5 | (u, c) rank, which orders them as their canonical
        // indices do. (Scanning the row for the kernel's grid sizes instead: 317,078 kernels of 128 points,
        // k = 15, 1,267 us against 741.)
        struct Head {
            float c;
            int i;
        };
        auto peek = [&](unsigned places, int B, float X, int base) -> Head {
            const int Bv = max(B, 1) - 1;  // (lanes without a triple have no places, and B* = 0)
            const int g = ct.rperm[Bv][(31 - __clz(places | 1u))];
            return {places ? __fmul_rn(X, ct.ipar[Bv][g]) : kInf, places ? base | (g << 5) : 0x7fffffff};
        };
        auto drop = [&](unsigned places) { return places & ~(0x80000000u >> __clz(places | 1u)); };

        // Merge: the warp repeatedly takes the smallest head and inserts it while it beats the k-th
        // entry. A lane's walk is in (cost, index) order unless two nearly equal
        // ipar values round to one cost, or X underflows; then (relaxed) equal
        // costs are walked on until a head costs more than the k-th entry.
        auto merge = [&](unsigned places, int B, float X, int base) {
            const bool relaxed = !ct.order_safe || __any_sync(kFull, places != 0u && !(X >= 0x1p-100f));
            Head h = peek(places, B, X, base);
            for (;;) {
                const unsigned mc = __reduce_min_sync(kFull, __float_as_uint(h.c));
                const float mcf = __uint_as_float(mc);
                const unsigned mi = __reduce_min_sync(kFull, h.c == mcf ? (unsigned)h.i : 0xffffffffu);
                if (mc >= 0x7f800000u || mcf > tau0 || mcf > tau_c) break;
                const bool enters = key_less(mcf, (int)mi, tau_c, tau_i);
                if (!enters && !relaxed) break;
                if (enters) warp_list_insert(lc, li, tau_c, tau_i, mcf, (int)mi, k, lane);
                if (h.c == mcf && h.i == (int)mi) {
                    places = drop(places);
                    h = peek(places, B, X, base);
                }
            }
        };

        {
            // ---- pre-pass over (T, U) pairs, lane = pair rank mod 32, carveouts inner.
            // Every grid size G of a triple costs X(T,U,C) * ipar(B*, G); a product by
            // X > 0 is monotone under round-to-nearest, so the triple's cheapest point
            // is exactly X * min_G ipar(B*, G). Each lane keeps the two smallest pair minima
            // (the smallest triple minimum over a (T, U) pair's carveouts) of its pairs, each
            // with its multiplicity (the pair's carveouts whose minimum equals it: the
            // carveouts of a pair often share B* and so their cost); tau0 is the smallest
            // value at which these entries, in increasing order, count k triples, and so
            // bounds the kernel's k-th best cost (k distinct triples each own a point
            // <= tau0). Each minimum is also stored at its triple rank (t rank * nUC +
            // u rank * nC + c rank), so that the carveouts of one (T, U) pair sit in
            // neighbouring lanes of the scan.
            const int nP = nT * nU;
            const int n_prow = (nP + 31) >> 5;
            const int n_blk = (nP * nC + 127) >> 7;  // blocks of 128 triples for the scan
            const float rcp_u = ct.rcpn[nU], rcp_c = ct.rcpn[nC], rcp_uc = ct.rcpn[nUC];
            {  // tail of the last block: no triple (NaN)
                const float nan = __int_as_float(0x7fc00000);
                *reinterpret_cast<float4*>(&w.key[((n_blk - 1) << 7) + 4 * lane]) = make_float4(nan, nan, nan, nan);
            }
            __syncwarp();
            float m0 = kInf, m1 = kInf;  // this lane's two smallest pair minima, ascending
            int c0 = 0, c1 = 0;          // their multiplicities
            // one body per carveout count, so that G_S stays in registers and a pair's
            // minima are stored with one vector store
            auto pairs = [&](auto nc_tag) {
                constexpr int NC = decltype(nc_tag)::value;
                int gs[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) gs[c] = w.gs[c];
                // pair pr = lane + 32 j = t_r nU + u_r, advanced by 32 pairs per step
                const int dq = small_div(32, rcp_u), dr = 32 - dq * nU;
                int t_r = small_div(lane, rcp_u), u_r = lane - t_r * nU;
                for (int j = 0; j < n_prow; ++j, t_r += dq, u_r += dr) {
                    const int pr = lane + (j << 5);
                    if (pr >= nP) break;
                    if (u_r >= nU) {
                        u_r -= nU;
                        ++t_r;
                    }
                    const int4 ti = w.tinfo[t_r];
                    const int wb = ti.x;
                    const float ln = __int_as_float(ti.y);
                    const float4 ui = w.uinfo[u_r];
                    const int gwr = block_limit(t_r, ti, u_r, ui);
                    const float cnm = ui.x, cmv = ui.y;
                    float key[NC];
                    float pm = kInf;
                    // branch-free: a triple without a valid configuration (B* = 0) reads
                    // hide[0] and iparmin[0] = NaN, so it is keyed NaN (never a
                    // candidate, not counted in the bound); W* = B* W_B <= W_mp <= kMaxW
                    // for a valid triple. X is finite (counts <= 2^40). Two carveouts at a
                    // time with packed FP32 operations, each rounded as the scalar ones.
#pragma unroll
                    for (int c = 0; c + 1 < NC; c += 2) {
                        const int B0 = min(gwr, gs[c]), B1 = min(gwr, gs[c + 1]);
                        const float2 X = mul2(fma2(make_float2(cmv, cmv), make_float2(ct.hide[B0 * wb], ct.hide[B1 * wb]),
                                                   make_float2(cnm, cnm)),
                                              make_float2(ln, ln));
                        const float2 kk = mul2(X, make_float2(w.iparmin[B0], w.iparmin[B1]));
                        key[c] = kk.x;
                        key[c + 1] = kk.y;
                        pm = fminf(pm, fminf(kk.x, kk.y));
                    }
                    if constexpr (NC & 1) {
                        const int B = min(gwr, gs[NC - 1]);
                        const float X = __fmul_rn(__fmaf_rn(cmv, ct.hide[B * wb], cnm), ln);
                        key[NC - 1] = __fmul_rn(X, w.iparmin[B]);
                        pm = fminf(pm, key[NC - 1]);
                    }
                    int mult = 0;
#pragma unroll
                    for (int c = 0; c < NC; ++c) mult += key[c] == pm ? 1 : 0;
                    {
                        const bool lt0 = pm < m0, lt1 = pm < m1;
                        m1 = lt0 ? m0 : (lt1 ? pm : m1);
                        c1 = lt0 ? c0 : (lt1 ? mult : c1);
                        m0 = lt0 ? pm : m0;
                        c0 = lt0 ? mult : c0;
                    }
                    float* krow = &w.key[pr * NC];
                    if constexpr (NC == 4) {
                        *reinterpret_cast<float4*>(krow) = make_float4(key[0], key[1], key[2], key[3]);
                    } else if constexpr (NC == 2) {
                        *reinterpret_cast<float2*>(krow) = make_float2(key[0], key[1]);
                    } else {
#pragma unroll
                        for (int c = 0; c < NC; ++c) krow[c] = key[c];
                    }
                }
            };
            switch (nC) {
                case 1: pairs(IntC<1>{}); break;
                case 2: pairs(IntC<2>{}); break;
                case 3: pairs(IntC<3>{}); break;
                default: pairs(IntC<4>{}); break;
            }
            __syncwarp();
            // entries in increasing order, equal ones at once, until they count k triples (a
            // finite entry counts at least one triple; +inf: fewer than k valid triples)
            for (int need = k;;) {
                const unsigned mb = __reduce_min_sync(kFull, __float_as_uint(m0));
                tau0 = __uint_as_float(mb);
                if (mb >= 0x7f800000u) break;
                const bool me = __float_as_uint(m0) == mb;  // the lanes whose smallest is taken
                need -= __reduce_add_sync(kFull, me ? c0 : 0);
                if (need <= 0) break;
                m0 = me ? m1 : m0;
                c0 = me ? c1 : c0;
                m1 = me ? kInf : m1;
                c1 = me ? 0 : c1;
            }

            // ---- candidates: the triples whose minimum does not exceed tau0 (every point
            // of the top-k belongs to one), four per lane and 128 per step. Their ranks
            // are compacted in place to the front of the key array: a slot written in
            // block b lies in blocks <= b, whose keys every lane has read before the
            // ballot.
            int n_cand = 0;
            for (int b = 0; b < n_blk; ++b) {
                const int t0 = (b << 7) + 4 * lane;  // this lane's four triples
                const float4 kv = *reinterpret_cast<const float4*>(&w.key[t0]);
                const unsigned m = (kv.x <= tau0 ? 1u : 0u) | (kv.y <= tau0 ? 2u : 0u) |
                                   (kv.z <= tau0 ? 4u : 0u) | (kv.w <= tau0 ? 8u : 0u);
                if (__ballot_sync(kFull, m != 0u) == 0u) continue;
                // in triple order: those of the lanes before, then this lane's
                int at = n_cand;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const unsigned bj = __ballot_sync(kFull, (m >> j) & 1u);
                    at += __popc(bj & below);
                    n_cand += __popc(bj);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if ((m >> j) & 1u) w.key[at++] = __int_as_float(t0 + j);
            }
            __syncwarp();

            // ---- selection: candidate triples 32 at a time, one per lane; each lane walks
            // its triple's grid sizes in increasing cost. The first batch starts from an
            // empty list, so its points, extracted in increasing cost, are appended at
            // list positions 0, 1, ... (a point that comes out of index order among equal
            // costs is inserted at its place instead); later batches merge into the list.
            for (int c0 = 0; c0 < n_cand; c0 += 32) {
                const bool has = c0 + lane < n_cand;
                int B = 0, base = 0;
                unsigned places = 0;
                float X = 0.0f;
                if (has) {
                    const int tri = __float_as_int(w.key[c0 + lane]);
                    const int t_r = small_div(tri, rcp_uc);
                    const int uc_r = tri - t_r * nUC;
                    const int u_r = small_div(uc_r, rcp_c);
                    const int c = uc_r - u_r * nC;
                    const int4 ti = w.tinfo[t_r];
                    const float4 ui = w.uinfo[u_r];
                    B = min(block_limit(t_r, ti, u_r, ui), w.gs[c]);
                    X = __fmul_rn(__fmaf_rn(ui.y, ct.hide[B * ti.x], ui.x), __int_as_float(ti.y));
                    base = t_r << 9 | uc_r;
                    places = g_dense ? all_places : w.places[B];
                }
                if (c0 > 0) {
                    merge(places, B, X, base);
                    continue;
                }
                Head h = peek(places, B, X, base);
                const bool relaxed = !ct.order_safe || __any_sync(kFull, has && !(X >= 0x1p-100f));
                if (!relaxed) {
                    // every lane's walk is in (cost, index) order: the r-th extraction is the
                    // r-th best of the batch (points above tau0 cannot be among the top k)
                    // (w.iparmin is free after the scan: list position r, then read by lane r)
                    float2* const list = reinterpret_cast<float2*>(w.iparmin);
                    int r = 0;
                    while (r < k) {
                        const unsigned mc = __reduce_min_sync(kFull, __float_as_uint(h.c));
                        const float mcf = __uint_as_float(mc);
                        if (mc >= 0x7f800000u || mcf > tau0) break;
                        const bool tie = h.c == mcf;
                        // every lane's next head, straight-line
                        const unsigned rest = drop(places);
                        const Head nx = peek(rest, B, X, base);
                        // Heads of the smallest cost whose index is below every equal-cost
                        // next head are the next points in (cost, index) order, all of them
                        // (each walk is in that order). Where their indices rise with the
                        // lane, as they mostly do (candidates are in triple order), the
                        // first ones go to list positions r.. at once.
                        const unsigned bound =
                            __reduce_min_sync(kFull, tie && nx.c == mcf ? (unsigned)nx.i : 0xffffffffu);
                        const bool elig = tie && (unsigned)h.i < bound;
                        const unsigned eb = __ballot_sync(kFull, elig), before = eb & below;
                        const int hprev = __shfl_sync(kFull, h.i, before ? 31 - __clz(before) : lane);
                        bool take;
                        if (__all_sync(kFull, !elig || !before || hprev < h.i)) {
                            const int to = r + __popc(before);
                            take = elig && to < k;
                            if (take) list[to] = make_float2(h.c, __int_as_float(h.i));
                            r += __popc(eb);
                        } else {
                            // indices out of lane order: one point, the lowest index
                            const unsigned mi = __reduce_min_sync(kFull, tie ? (unsigned)h.i : 0xffffffffu);
                            take = tie && h.i == (int)mi;
                            if (take) list[r] = make_float2(h.c, __int_as_float(h.i));
                            ++r;
                        }
                        if (take) h = nx;
                        places = take ? rest : places;
                    }
                    __syncwarp();
                    if (lane < min(r, k)) {
                        const float2 e = list[lane];
                        lc = e.x;
                        li = __float_as_int(e.y);
                    }
                    tau_c = __shfl_sync(kFull, lc, k - 1);
                    tau_i = __shfl_sync(kFull, li, k - 1);
                    continue;
                }
                int cnt = 0;  // list entries so far; (prev_c, prev_i) is the largest
                float prev_c = 0.0f;
                int prev_i = -1;
                for (;;) {
                    const unsigned mc = __reduce_min_sync(kFull, __float_as_uint(h.c));
                    const float mcf = __uint_as_float(mc);
                    if (mc >= 0x7f800000u || mcf > tau0 || mcf > tau_c) break;
                    const unsigned mi = __reduce_min_sync(kFull, h.c == mcf ? (unsigned)h.i : 0xffffffffu);
                    if (cnt < k && (cnt == 0 || key_less(prev_c, prev_i, mcf, (int)mi))) {
                        if (lane == cnt) {  // in order: append
                            lc = mcf;
                            li = (int)mi;
                        }
                        prev_c = mcf;
                        prev_i = (int)mi;
                        if (++cnt == k) {
                            tau_c = __shfl_sync(kFull, lc, k - 1);
                            tau_i = __shfl_sync(kFull, li, k - 1);
                        }
                    } else if (key_less(mcf, (int)mi, tau_c, tau_i)) {
                        // out of index order among equal costs: insert at its place
                        warp_list_insert(lc, li, tau_c, tau_i, mcf, (int)mi, k, lane);
                        if (cnt < k && ++cnt == k) {
                            tau_c = __shfl_sync(kFull, lc, k - 1);
                            tau_i = __shfl_sync(kFull, li, k - 1);
                        }
                    }
                    if (h.c == mcf && h.i == (int)mi) {
                        places = drop(places);
                        h = peek(places, B, X, base);
                    }
                }
            }
        }
        if (lane < k) {
            const int g = (li >> 5) & 15;  // the canonical index of the numbered point
            const int at = (li >> 9) * g_stride + __popc(gm & ((1u << g) - 1u)) * nUC + (li & 31);
            topk_idx[kid * k + lane] = li < 0 ? -1 : at;
            topk_cost[kid * k + lane] = lc;
        }
        __syncwarp();  // the warp's tables are rewritten for the next descriptor
        if (EMIT) {
            // the tables stay for the emitting pass, the ipar rows in the place of the keys; the points of a small
            // space are written at once
            const bool small = nT * g_stride <= kEmitAlone;
            if (lane < kMaxB)
                for (int j = 0; j < nG; ++j) w.iparc[lane][j] = ct.ipar[lane][w.gpos[j]];
            if (lane == 0) {
                w.nT = small ? 0 : nT;
                w.nG = nG;
                w.nU = nU;
                w.nC = nC;
                w.simple = simple;
                w.off = pt_off[kid];
            }
            __syncwarp();
            if (small) emit_points(ct, w, w.tri, 0, nT, lane, pt_b, pt_w, pt_c);
        }
    };

    if constexpr (EMIT) {
        // A CTA takes `group` descriptors at a time (from the grid's queue), a warp ranks each, and then all its
        // warps write each one's points, an eighth of the thread counts each: the spaces' sizes differ, and a warp
        // by itself needs 25 us for the points of a full one. Towards the end of the descriptors the groups shrink, to
        // as few as have about 16,384 points (by the mean of the offsets), so that no CTA is left with eight large
        // spaces. (20,000 uneven kernels, 114 M points: 534 us with a warp per descriptor, lanes on triples and each
        // lane writing its grid sizes nUC points apart; 316 with the points written in order; 280 shared by the CTA;
        // 253 with shrinking groups, the HBM floor being 201; 6,000 dense ones: 226 -> 181, 0.96 of the HBM rate.)
        __shared__ long long next;
        __shared__ int next_size;
        const int warp = threadIdx.x >> 5;
        int least = 1;
        if (threadIdx.x == 0) {
            const int64_t mean = n_k > 1 ? max((int64_t)1, (pt_off[n_k - 1] - pt_off[0]) / (n_k - 1)) : 1;
            least = (int)max((int64_t)1, min((int64_t)kWarps, 16384 / mean));
        }
        int size = p.group;
        for (int64_t g = (int64_t)blockIdx.x * size; g < n_k;) {
            if (threadIdx.x == 0) {
                const int64_t even = (n_k - g) / (4 * (int64_t)gridDim.x);
                next_size = min(p.group, (int)max((int64_t)least, min((int64_t)kWarps, even)));
                next = (long long)gridDim.x * p.group + (long long)atomicAdd(queue, (unsigned long long)next_size);
            }
            const int64_t kid = g + warp;
            if (lane == 0) w.nT = 0;
            __syncwarp();
            if (warp < size && kid < n_k) rank(kid, __ldg(descs + kid * 4 + (lane & 3)));
            __syncthreads();
            for (int i = 0; i < size; ++i) {
                const WarpTables& t = wts[i];
                emit_points(ct, t, w.tri, warp * t.nT / kWarps, (warp + 1) * t.nT / kWarps, lane, pt_b, pt_w, pt_c);
            }
            g = next;
            size = next_size;
            __syncthreads();  // the tables and `next` are rewritten
        }
        return;
    }

    int64_t kid, q_end = 0;
    if (p.chunk == 0) {
        kid = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    } else {
        grab();
        kid = grabbed_kid();
        q_end = min(kid + p.chunk, n_k);
    }
    if (kid < n_k) grab();
    // lanes 0..3 hold the four 16-byte words of the descriptor (lane & 3)
    int4 v = kid < n_k ? __ldg(descs + kid * 4 + (lane & 3)) : make_int4(0, 0, 0, 0);
    while (kid < n_k) {
        int64_t nk;
        if (kid + 1 < q_end) {  // (q_end stays 0 without the grid's queue)
            nk = kid + 1;
        } else {
            nk = grabbed_kid();
            if (p.chunk) q_end = min(nk + p.chunk, n_k);
            if (nk < n_k) grab();
        }
        const int4 v_next = nk < n_k ? __ldg(descs + nk * 4 + (lane & 3)) : make_int4(0, 0, 0, 0);
        rank(kid, v);
        kid = nk;
        v = v_next;
    }
    // A row is complete only after the row before it. One CTA waits: if all did, those that find the queue empty would
    // keep their places from the rows after (9,800 dense kernels against six rows, 16 per grab: 658 us, now 288).
    if (blockIdx.x == 0) pdl::grid_dep_wait();
}

// ---- thread-per-kernel schedule ---------------------------------------------
//
// One thread evaluates one kernel descriptor: per-unroll tables in shared
// memory (one column per thread), per-carveout limits packed in a register,
// then a bound pre-pass and the main pass over (T, U, C) triples with every
// grid size's cost computed. The thread keeps a sorted register list of its k
// best (cost, index); no warp collectives are involved, so kernels of any
// space size run without per-kernel warp overhead.

constexpr int kThreadsT = 128;

template <int KMAX>
__device__ __forceinline__ void tlist_insert(float (&lc)[KMAX], int (&li)[KMAX], float c, int i)
{
#pragma unroll
    for (int j = KMAX - 1; j > 0; --j) {
        const bool shift = key_less(c, i, lc[j - 1], li[j - 1]);
        const bool here = !shift && key_less(c, i, lc[j], li[j]);
        const float nc = shift ? lc[j - 1] : (here ? c : lc[j]);
        const int ni = shift ? li[j - 1] : (here ? i : li[j]);
        lc[j] = nc;
        li[j] = ni;
    }
    if (key_less(c, i, lc[0], li[0])) {
        lc[0] = c;
        li[0] = i;
    }
}

template <int KMAX, typename V>
__device__ __forceinline__ V list_kth(const V (&l)[KMAX], int k)
{
    // Select chain (not l[k - 1], which would force the list into local memory).
    V t = l[KMAX - 1];
#pragma unroll
    for (int j = KMAX - 2; j >= 0; --j) t = (j >= k - 1) ? l[j] : t;
    return t;
}

// Sorted insert of a value into an ascending list, dropping the largest.
template <int KMAX>
__device__ __forceinline__ void value_insert(float (&l)[KMAX], float v)
{
#pragma unroll
    for (int j = 0; j < KMAX; ++j) {
        const float lo = fminf(l[j], v);
        v = fmaxf(l[j], v);
        l[j] = lo;
    }
}

// 80 registers for six CTAs per SM; 84, which the compiler takes when it may, leave five (100,000 kernels of 128
// points, k = 5: 289 us instead of 190).
template <int KMAX>
__global__ void __maxnreg__(KMAX > 8 ? 128 : 80)
    tune_eval_thread_kernel(const __grid_constant__ EvalParams p, const int4* __restrict__ descs,
                            int32_t* __restrict__ topk_idx, float* __restrict__ topk_cost,
                            int* __restrict__ status)
{
    __shared__ CtaTables ct;
    __shared__ float4 utab[8][kThreadsT];  // per unroll position: C_nm, C_m, R, warps | wbmax << 8
    const tune_arch& a = p.a;
    copy_cta_tables(p.tab, ct);
    __syncthreads();

    const tune_axes& x = p.x;
    const float kInf = __int_as_float(0x7f800000);
    const int k = p.k;
    const int tid = threadIdx.x;
    const uint32_t g_all = (1u << x.n_g) - 1u;

    for (int64_t kid = (int64_t)blockIdx.x * kThreadsT + tid; kid < p.n_kernels;
         kid += (int64_t)gridDim.x * kThreadsT) {
        int4 vw[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) vw[q] = __ldg(descs + kid * 4 + q);
        Desc kd;
        unpack(vw, kd);
        const uint32_t tm = kd.tm, gm = kd.gm, um = kd.um, cm = kd.cm;
        const bool bad = desc_bad(kd, x);
        const int nT = __popc(tm), nG = __popc(gm), nU = __popc(um), nC = __popc(cm);
        if (bad || nT * nG * nU * nC == 0) {
            if (bad) atomicOr(status, tune::kStatusInvalid);
            for (int j = 0; j < k; ++j) {
                topk_idx[kid * k + j] = -1;
                topk_cost[kid * k + j] = kInf;
            }
            continue;
        }
        const int nUC = nU * nC;
        const int g_stride = nG * nUC;
        const bool g_dense = gm == g_all;

        // ---- per-unroll and per-carveout tables
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if ((um >> u) & 1u) {
                const int U = x.u[u];
                const int R = kd.r0 + 4 * (U - 1);
                float cnm, cmv;
                unit_costs(kd.n, kd.d, U, ct.rcp, a.work_scale, cnm, cmv);
                int warps, wbmax;
                reg_params(a, R, warps, wbmax);
                utab[u][tid] = make_float4(cnm, cmv, __int_as_float(R),
                                           __int_as_float(warps | (min(wbmax, 255) << 8)));
            }
        }
        uint32_t gsp = 0;  // G_S per carveout position, one byte each
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if ((cm >> c) & 1u) gsp |= (uint32_t)min(smem_blocks(a, kd.s0, x.c[c]), 255) << (8 * c);

        // ---- loop nest over the triples in canonical (T, U, C) order; body(B, W, X, base)
        auto for_triples = [&](auto&& body) {
            int t_r = 0;
            for (uint32_t tb = tm; tb; tb &= tb - 1u, ++t_r) {
                const int tp = __ffs(tb) - 1;
                const int wb = ct.wb[tp], gw = ct.gw[tp];
                const float ln = ct.lane[tp];
                int u_r = 0;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (!((um >> u) & 1u)) continue;
                    const float4 ut = utab[u][tid];
                    const int wr = __float_as_int(ut.w);
                    const int bu = min(gw, reg_blocks(a, ct, __float_as_int(ut.z), wb, tp, wr & 0xff, wr >> 8));
                    int c_r = 0;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (!((cm >> c) & 1u)) continue;
                        const int B = min(bu, (int)((gsp >> (8 * c)) & 0xffu));
                        if (B > 0) {
                            const int W = B * wb;
                            const float X = __fmul_rn(__fmaf_rn(ut.y, ct.hide[W], ut.x), ln);
                            body(B, X, t_r * g_stride + u_r * nC + c_r);
                        }
                        ++c_r;
                    }
                    ++u_r;
                }
            }
        };

        // ---- pre-pass: tau0 = k-th smallest triple minimum (k distinct triples each
        // own a point of cost <= tau0, so the k-th best point is <= tau0).
        float tk[KMAX];
#pragma unroll
        for (int j = 0; j < KMAX; ++j) tk[j] = kInf;
        float tau0 = kInf;
        for_triples([&](int B, float X, int) {
            float mn;
            if (g_dense) {
                mn = ct.iparmin[B - 1];
            } else {
                mn = kInf;
                for (uint32_t gb = gm; gb; gb &= gb - 1u) mn = fminf(mn, ct.ipar[B - 1][__ffs(gb) - 1]);
            }
            const float m = __fmul_rn(X, mn);
            if (m < tau0) {
                value_insert<KMAX>(tk, m);
                tau0 = list_kth<KMAX>(tk, k);
            }
        });

        // ---- main pass: every point's cost, folded into its triple's minimum;
        // points that can still enter the list are inserted exactly.
        float lc[KMAX];
        int li[KMAX];
#pragma unroll
        for (int j = 0; j < KMAX; ++j) {
            lc[j] = kInf;
            li[j] = -1;
        }
        float thr_c = kInf;
        int thr_i = -1;
        for_triples([&](int B, float X, int base) {
            if (g_dense) {
                // the triple's cheapest point (a product by X > 0 keeps the order of ipar)
                const float cmin = __fmul_rn(X, ct.iparmin[B - 1]);
                if (cmin <= fminf(thr_c, tau0)) {
                    // grid sizes in increasing cost: the order of ipar(B*, G) over G
#pragma unroll 1
                    for (int r = 0; r < x.n_g; ++r) {
                        const int g = ct.rperm[B - 1][15 - r];
                        const float cg = __fmul_rn(X, ct.ipar[B - 1][g]);
                        if (cg > fminf(thr_c, tau0)) break;
                        const int idx = base + g * nUC;
                        if (key_less(cg, idx, thr_c, thr_i)) {
                            tlist_insert<KMAX>(lc, li, cg, idx);
                            thr_c = list_kth<KMAX>(lc, k);
                            thr_i = list_kth<KMAX>(li, k);
                        }
                    }
                }
            } else {
                int g_r = 0;
                for (uint32_t gb = gm; gb; gb &= gb - 1u, ++g_r) {
                    const float cg = __fmul_rn(X, ct.ipar[B - 1][__ffs(gb) - 1]);
                    if (cg <= fminf(thr_c, tau0)) {
                        const int idx = base + g_r * nUC;
                        if (key_less(cg, idx, thr_c, thr_i)) {
                            tlist_insert<KMAX>(lc, li, cg, idx);
                            thr_c = list_kth<KMAX>(lc, k);
                            thr_i = list_kth<KMAX>(li, k);
                        }
                    }
                }
            }
        });
#pragma unroll
        for (int j = 0; j < KMAX; ++j) {
            if (j < k) {
                topk_idx[kid * k + j] = li[j];
                topk_cost[kid * k + j] = lc[j];
            }
        }
    }
}

template <int KMAX>
int launch_thread(const EvalParams& p, const tune_kernel_desc* descs, int32_t* ti, float* tc, int* status,
                  cudaStream_t s)
{
    auto kern = tune_eval_thread_kernel<KMAX>;
    static std::atomic<int> per_sm_cache[tune::kMaxDevices];
    int per_sm = 0;
    int rc = tune::blocks_per_sm(per_sm_cache, reinterpret_cast<const void*>(kern), kThreadsT, &per_sm);
    if (rc) return rc;
    const int sms = tune::device_sm_count();
    if (sms <= 0) return tune::fail(TUNE_ECUDA, "tune_eval: cannot query the SM count");
    const int64_t need = (p.n_kernels + kThreadsT - 1) / kThreadsT;
    const int64_t cap = (int64_t)sms * per_sm;
    const int grid = (int)(need < cap ? need : cap);
    EvalParams q = p;
    tune::eval_tables(q.a, q.x, q.tab);
    kern<<<grid, kThreadsT, 0, s>>>(q, reinterpret_cast<const int4*>(descs), ti, tc, status);
    TUNE_CUDA_TRY(cudaGetLastError(), "tune_eval: kernel launch");
    return TUNE_OK;
}

// Queue counter `i` of a workspace header: the 8-byte words after the status word, wherever in memory the caller's
// workspace begins (the ranking by default needs the status word's alignment only, the emitting pass always a queue).
unsigned long long* queue_word(int* status, int i)
{
    return reinterpret_cast<unsigned long long*>((reinterpret_cast<uintptr_t>(status + 1) + 7) & ~uintptr_t(7)) + i;
}

// Row `row` of the `rows` of a sweep. Rows after the first may start while the one before them still runs.
template <bool EMIT>
int launch(const EvalParams& p, const tune_kernel_desc* descs, int32_t* ti, float* tc, int32_t* pb, int32_t* pw,
           float* pc, const int64_t* po, int* status, cudaStream_t s, int ctas_per_sm = 0,
           unsigned long long* queue = nullptr, int row = 0, int rows = 1)
{
    auto kern = tune_eval_kernel<EMIT>;
    static std::atomic<int> per_sm_cache[tune::kMaxDevices];
    int per_sm = 0;
    int rc = tune::blocks_per_sm(per_sm_cache, reinterpret_cast<const void*>(kern), kThreads, &per_sm);
    if (rc) return rc;
    const int sms = tune::device_sm_count();
    if (sms <= 0) return tune::fail(TUNE_ECUDA, "tune_eval: cannot query the SM count");
    const int64_t need = (p.n_kernels + kWarps - 1) / kWarps;
    int64_t cap = (int64_t)sms * (ctas_per_sm > 0 ? min(ctas_per_sm, per_sm) : per_sm);
    // Where a row has few descriptors per warp of a full grid, the rows share the chip's places side by side instead:
    // up to three per warp (12,000 dense kernels against six rows: 148 us, row by row 151; 20,000, 4.1 per warp: 234
    // against 223), with a work queue up to four (15,000 uneven ones against eight rows: 198 us against 233; 30,000
    // dense ones against six: 5 % slower). No more CTAs than places: with four above the 608, six rows of 9,000 dense
    // kernels took 145 us, now 120.
    if (rows > 1 && need < (p.chunk ? 4 : 3) * cap) cap = std::max<int64_t>(1, cap / rows);
    const int grid = (int)std::min(EMIT ? p.n_kernels : need, cap);
    // By default the first queue counter of the zeroed workspace header.
    if (!queue) queue = queue_word(status, 0);
    EvalParams q = p;
    q.next_row = row + 1 < rows;
    // A sweep's grabs: about four per warp at least, else the rows end with a few warps that walk long chunks (9,800
    // dense kernels against six rows, 16 per grab: 288 us, now 130).
    if (rows > 1 && q.chunk > 1) q.chunk = (int)std::max<int64_t>(1, std::min<int64_t>(q.chunk, p.n_kernels / (4 * kWarps * (int64_t)grid)));
    // emitting: as many descriptors at a time, up to one per warp, as leave each CTA about three turns (the queue
    // evens out spaces of different sizes), or one turn where a single array is written: ranking then takes longer than
    // the stores, and wants all warps (3,000 dense kernels, B* alone: 62 us with three turns, 49 with one, 57 with a
    // warp per descriptor; all three arrays 101 us with three, 110 with one, 123).
    const int64_t most = (pb != nullptr) + (pw != nullptr) + (pc != nullptr) > 1 ? p.n_kernels / (3 * cap) : (p.n_kernels + cap - 1) / cap;
    q.group = (int)std::max<int64_t>(1, std::min<int64_t>(kWarps, most));
    tune::eval_tables(q.a, q.x, q.tab);
    const int4* d = reinterpret_cast<const int4*>(descs);
    if (row > 0)
        TUNE_CUDA_TRY(pdl::launch_dep(kern, dim3(grid), dim3(kThreads), 0, s, q, d, ti, tc, pb, pw, pc, po, status, queue),
                      "tune_eval: kernel launch");
    else
        kern<<<grid, kThreads, 0, s>>>(q, d, ti, tc, pb, pw, pc, po, status, queue);
    TUNE_CUDA_TRY(cudaGetLastError(), "tune_eval: kernel launch");
    return TUNE_OK;
}

int validate(const tune_arch* a, const tune_axes* x, int32_t k)
{
    if (k < 1 || k > 16) return tune::fail(TUNE_EINVAL, "k = %d outside [1, 16]", k);
    return tune::validate_inputs(a, x);
}

}  // namespace

namespace tune {

int validate_inputs(const tune_arch* a, const tune_axes* x)
{
    if (!a || !x) return fail(TUNE_EINVAL, "arch and axes must be non-NULL host pointers");
    if (a->warp_size != 32) return fail(TUNE_EINVAL, "warp_size must be 32");
    if (a->n_sm < 1 || a->max_threads_block < 1 || a->max_warps_sm < 1 || a->max_warps_sm > kMaxW ||
        a->max_blocks_sm < 1 || a->max_blocks_sm > kMaxB)
        return fail(TUNE_EINVAL, "arch: n_sm, max_threads_block, max_warps_sm (<=64) or "
                                 "max_blocks_sm (<=32) out of range");
    if (a->regs_sm < 1 || a->regs_block_max < 1 || a->regs_thread_max < 1 ||
        a->regs_thread_max > 65536 || a->reg_alloc_unit < 1 || a->reg_alloc_unit > 65536 ||
        a->warp_alloc_gran < 1 || (a->reg_alloc_mode != 0 && a->reg_alloc_mode != 1))
        return fail(TUNE_EINVAL, "arch: register fields out of range");
    if (a->smem_block_max < 0 || a->smem_block_max > (1 << 24) || a->smem_reserved_block < 0 ||
        a->smem_reserved_block > (1 << 24) || a->smem_alloc_unit < 1 || a->smem_alloc_unit > (1 << 20) ||
        a->n_smem_caps < 1 || a->n_smem_caps > 16)
        return fail(TUNE_EINVAL, "arch: shared-memory fields out of range");
    for (int i = 0; i < a->n_smem_caps; ++i)
        if (a->smem_caps[i] < 0 || (i > 0 && a->smem_caps[i] < a->smem_caps[i - 1]) ||
            a->smem_caps[i] > (1 << 24))
            return fail(TUNE_EINVAL, "arch: smem_caps must be ascending, in [0, 16 MB]");
    for (int c = 0; c < TUNE_NCLASS; ++c)
        if (!(a->ipc[c] >= 0x1p-16f) || !isfinite(a->ipc[c]))
            return fail(TUNE_EINVAL, "arch: ipc[%d] must be finite and >= 2^-16", c);
    if (a->w_sat < 1 || a->w_sat > (1 << 20) || a->work_scale < 1 || a->work_scale > (1 << 24))
        return fail(TUNE_EINVAL, "arch: w_sat or work_scale out of range");
    if (x->n_t < 1 || x->n_t > 32 || x->n_g < 1 || x->n_g > 16 || x->n_u < 1 || x->n_u > 8 ||
        x->n_c < 1 || x->n_c > 4)
        return fail(TUNE_EINVAL, "axes: lengths out of range");
    for (int i = 0; i < x->n_t; ++i)
        if (x->t[i] < 1 || x->t[i] > 4096) return fail(TUNE_EINVAL, "axes: t[%d] outside [1, 4096]", i);
    for (int i = 0; i < x->n_g; ++i) {
        if (x->g[i] < 1 || (int64_t)a->n_sm * x->g[i] >= (1 << 24) ||
            (int64_t)x->g[i] + (int64_t)a->n_sm * a->max_blocks_sm >= (1 << 24))
            return fail(TUNE_EINVAL, "axes: g[%d] must be >= 1 with n_sm * g < 2^24", i);
    }
    for (int i = 0; i < x->n_u; ++i)
        if (x->u[i] < 1 || x->u[i] > 64) return fail(TUNE_EINVAL, "axes: u[%d] outside [1, 64]", i);
    for (int i = 0; i < x->n_c; ++i)
        if (x->c[i] < 0 || x->c[i] > 100) return fail(TUNE_EINVAL, "axes: c[%d] outside [0, 100]", i);
    return TUNE_OK;
}

}  // namespace tune

extern "C" int tune_eval(const tune_arch* arch, const tune_axes* axes, const tune_kernel_desc* descs,
                         int64_t n_kernels, int32_t k, uint32_t flags, int32_t* topk_idx,
                         float* topk_cost, int32_t* pt_blocks, int32_t* pt_warps, float* pt_cost,
                         const int64_t* pt_offsets, void* workspace, size_t ws_bytes,
                         tune_stream_t stream)
{
    tune::clear_error();
    int rc = validate(arch, axes, k);
    if (rc) return rc;
    if (n_kernels < 0) return tune::fail(TUNE_EINVAL, "n_kernels < 0");
    if (!workspace) return tune::fail(TUNE_EINVAL, "workspace is NULL");
    if (ws_bytes < tune_workspace_bytes(TUNE_CALL_EVAL, n_kernels, k))
        return tune::fail(TUNE_ENOMEM, "workspace of %zu bytes is smaller than %zu", ws_bytes,
                          tune_workspace_bytes(TUNE_CALL_EVAL, n_kernels, k));
    if (n_kernels > 0 && (!descs || !topk_idx || !topk_cost))
        return tune::fail(TUNE_EINVAL, "descs, topk_idx and topk_cost must be non-NULL");
    if ((reinterpret_cast<uintptr_t>(descs) & 15) != 0)
        return tune::fail(TUNE_EINVAL, "descs must be 16-byte aligned");
    if (flags & ~(TUNE_EMIT_POINTS | TUNE_SCHED_WARP | TUNE_SCHED_THREAD | 0xff00u))
        return tune::fail(TUNE_EINVAL, "unknown flags 0x%x", flags);
    const int chunk_code = (int)((flags >> 8) & 0xfu);
    if (chunk_code > 15) return tune::fail(TUNE_EINVAL, "bad chunk code");
    const int chunk = chunk_code == 0 ? 0 : (1 << (chunk_code - 1));
    const int ctas_per_sm = (int)((flags >> 12) & 0xfu);
    const bool emit = (flags & TUNE_EMIT_POINTS) != 0;
    if (emit && !pt_offsets) return tune::fail(TUNE_EINVAL, "TUNE_EMIT_POINTS needs pt_offsets");
    if ((flags & TUNE_SCHED_WARP) && (flags & TUNE_SCHED_THREAD))
        return tune::fail(TUNE_EINVAL, "TUNE_SCHED_WARP and TUNE_SCHED_THREAD are exclusive");
    if (emit && (flags & TUNE_SCHED_THREAD))
        return tune::fail(TUNE_EINVAL, "TUNE_EMIT_POINTS runs on the warp schedule only");
    const bool thread_sched = (flags & TUNE_SCHED_THREAD) != 0;

    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int* status = static_cast<int*>(workspace);
    TUNE_CUDA_TRY(cudaMemsetAsync(workspace, 0, tune::kWorkspaceHeader, s), "tune_eval: status reset");
    if (n_kernels == 0) return TUNE_OK;

    EvalParams p;
    p.a = *arch;
    p.x = *axes;
    p.n_kernels = n_kernels;
    p.k = k;
    p.chunk = chunk;
    if (thread_sched)
        return k <= 8 ? launch_thread<8>(p, descs, topk_idx, topk_cost, status, s)
                      : launch_thread<16>(p, descs, topk_idx, topk_cost, status, s);
    return emit ? launch<true>(p, descs, topk_idx, topk_cost, pt_blocks, pt_warps, pt_cost, pt_offsets,
                               status, s, ctas_per_sm)
                : launch<false>(p, descs, topk_idx, topk_cost, nullptr, nullptr, nullptr, nullptr, status,
                                s, ctas_per_sm);
}

// ---------------------------------------------------------------------------
// tune_eval_noalloc: the same evaluation for callers that cannot hand the
// library a workspace. Some hosts own every byte of device memory (a serving
// runtime or a framework allocator that gives plugins no way to ask for a
// buffer), and some run under a device-memory budget fixed at start-up that
// must not grow afterwards; neither can call cudaMalloc on the library's
// behalf. This entry point keeps its scratch in the file-scope array below
// instead, which every GPU that loads the library holds until the process
// exits, and allocates nothing itself.
// ---------------------------------------------------------------------------

namespace {

constexpr size_t kNoallocScratchBytes = 4096;  // stated maximum scratch for one call

// Scratch of tune_eval_noalloc: a header (status word and the emitting pass's queue) per call under way. Calls
// that shared one would take descriptor groups from each other's queue and leave points unwritten.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];
constexpr int kNoallocHeaders = (int)(kNoallocScratchBytes / tune::kWorkspaceHeader);
static_assert(kNoallocHeaders <= 32, "a bit per header");

struct NoallocDevice {
    std::mutex mu;
    std::condition_variable freed;
    char* base = nullptr;  // device address of the array, looked up once
    uint32_t busy = 0;     // headers in use
};
NoallocDevice g_noalloc[tune::kMaxDevices];

// One of the current device's headers, the caller's until the object goes (waits while all are taken).
class NoallocHeader {
public:
    ~NoallocHeader()
    {
        if (!ptr_) return;
        std::lock_guard<std::mutex> lock(dev_->mu);
        dev_->busy &= ~(1u << slot_);
        dev_->freed.notify_one();
    }
    // (Host code must not use the array's symbol itself: on the host it names a stand-in object, not device memory.)
    int take(void** out)
    {
        int dev = 0;
        TUNE_CUDA_TRY(cudaGetDevice(&dev), "tune_eval_noalloc: cudaGetDevice");
        if (dev < 0 || dev >= tune::kMaxDevices) return tune::fail(TUNE_EUNSUPPORTED, "device ordinal %d too large", dev);
        dev_ = &g_noalloc[dev];
        std::unique_lock<std::mutex> lock(dev_->mu);
        if (!dev_->base) {
            void* p = nullptr;
            TUNE_CUDA_TRY(cudaGetSymbolAddress(&p, g_noalloc_scratch), "tune_eval_noalloc: cudaGetSymbolAddress");
            dev_->base = static_cast<char*>(p);
        }
        constexpr uint32_t all = (uint32_t)((1ull << kNoallocHeaders) - 1);
        dev_->freed.wait(lock, [&] { return dev_->busy != all; });
        slot_ = __builtin_ctz(~dev_->busy);
        dev_->busy |= 1u << slot_;
        ptr_ = *out = dev_->base + slot_ * tune::kWorkspaceHeader;
        return TUNE_OK;
    }

private:
    NoallocDevice* dev_ = nullptr;
    void* ptr_ = nullptr;
    int slot_ = 0;
};

// The call on its header: everything that uses it is complete when this returns TUNE_OK.
int noalloc_call(void* scratch, EvalParams& p, const tune_kernel_desc* descs, bool emit, int32_t* topk_idx, float* topk_cost,
                 int32_t* pt_blocks, int32_t* pt_warps, float* pt_cost, const int64_t* pt_offsets, cudaStream_t s)
{
    // The array keeps earlier calls' contents: clear the status word and counters.
    TUNE_CUDA_TRY(cudaMemsetAsync(scratch, 0, tune::kWorkspaceHeader, s), "tune_eval_noalloc: scratch reset");
    if (p.n_kernels > 0) {
        int* status = static_cast<int*>(scratch);
        const int rc = emit ? launch<true>(p, descs, topk_idx, topk_cost, pt_blocks, pt_warps, pt_cost, pt_offsets, status, s)
                            : launch<false>(p, descs, topk_idx, topk_cost, nullptr, nullptr, nullptr, nullptr, status, s);
        if (rc) return rc;
    }
    // Report what the kernel found: wait for the stream and read the status word.
    int st = 0;
    TUNE_CUDA_TRY(cudaMemcpyAsync(&st, scratch, sizeof(int), cudaMemcpyDeviceToHost, s),
                  "tune_eval_noalloc: status read");
    TUNE_CUDA_TRY(cudaStreamSynchronize(s), "tune_eval_noalloc: cudaStreamSynchronize");
    if (st & tune::kStatusTimeout) return tune::fail(TUNE_ETIMEOUT, "a bounded device-side wait gave up");
    if (st & tune::kStatusInvalid)
        return tune::fail(TUNE_EINVAL, "a descriptor was malformed (mask outside the axes, negative "
                                       "count, register or shared-memory field)");
    return TUNE_OK;
}

}  // namespace

extern "C" int tune_eval_noalloc(const tune_arch* arch, const tune_axes* axes,
                                 const tune_kernel_desc* descs, int64_t n_kernels, int32_t k,
                                 uint32_t flags, int32_t* topk_idx, float* topk_cost,
                                 int32_t* pt_blocks, int32_t* pt_warps, float* pt_cost,
                                 const int64_t* pt_offsets, tune_stream_t stream)
{
    tune::clear_error();
    int rc = validate(arch, axes, k);
    if (rc) return rc;
    if (n_kernels < 0) return tune::fail(TUNE_EINVAL, "n_kernels < 0");
    const size_t need = tune_workspace_bytes(TUNE_CALL_EVAL, n_kernels, k);
    if (need > kNoallocScratchBytes)
        return tune::fail(TUNE_ENOMEM,
                          "tune_eval_noalloc: this call needs %zu bytes of scratch, more than the "
                          "%zu-byte static area; use tune_eval with a workspace",
                          need, kNoallocScratchBytes);
    if (n_kernels > 0 && (!descs || !topk_idx || !topk_cost))
        return tune::fail(TUNE_EINVAL, "descs, topk_idx and topk_cost must be non-NULL");
    if ((reinterpret_cast<uintptr_t>(descs) & 15) != 0)
        return tune::fail(TUNE_EINVAL, "descs must be 16-byte aligned");
    if (flags & ~TUNE_EMIT_POINTS) return tune::fail(TUNE_EINVAL, "unknown flags 0x%x", flags);
    const bool emit = (flags & TUNE_EMIT_POINTS) != 0;
    if (emit && !pt_offsets) return tune::fail(TUNE_EINVAL, "TUNE_EMIT_POINTS needs pt_offsets");

    NoallocHeader header;
    void* scratch = nullptr;
    rc = header.take(&scratch);
    if (rc) return rc;
    EvalParams p;
    p.a = *arch;
    p.x = *axes;
    p.n_kernels = n_kernels;
    p.k = k;
    p.chunk = 0;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    rc = noalloc_call(scratch, p, descs, emit, topk_idx, topk_cost, pt_blocks, pt_warps, pt_cost, pt_offsets, s);
    if (rc) cudaStreamSynchronize(s);  // the header goes to the next call with nothing of this one under way
    return rc;
}

// ---------------------------------------------------------------------------
// tune_eval_archs: the same ranking for every kernel against several
// architecture rows.
// ---------------------------------------------------------------------------
extern "C" int tune_eval_archs(const tune_arch* archs, int32_t n_arch, const tune_axes* axes,
                               const tune_kernel_desc* descs, int64_t n_kernels, int32_t k, uint32_t flags,
                               int32_t* topk_idx, float* topk_cost, void* workspace, size_t ws_bytes,
                               tune_stream_t stream)
{
    tune::clear_error();
    if (!archs || n_arch < 1 || n_arch > kMaxArch)
        return tune::fail(TUNE_EINVAL, "n_arch = %d outside [1, %d] or archs NULL", n_arch, kMaxArch);
    for (int i = 0; i < n_arch; ++i) {
        int rc = validate(&archs[i], axes, k);
        if (rc) return rc;
    }
    if (n_kernels < 0) return tune::fail(TUNE_EINVAL, "n_kernels < 0");
    if (!workspace || ws_bytes < tune::kWorkspaceHeader)
        return tune::fail(TUNE_ENOMEM, "workspace smaller than %d bytes", tune::kWorkspaceHeader);
    if (n_kernels > 0 && (!descs || !topk_idx || !topk_cost))
        return tune::fail(TUNE_EINVAL, "descs, topk_idx and topk_cost must be non-NULL");
    if ((reinterpret_cast<uintptr_t>(descs) & 15) != 0)
        return tune::fail(TUNE_EINVAL, "descs must be 16-byte aligned");
    if (flags & ~(TUNE_SCHED_WARP | 0xff00u))
        return tune::fail(TUNE_EINVAL, "flags 0x%x: only TUNE_SCHED_WARP and its chunk/CTA fields", flags);
    const int chunk_code = (int)((flags >> 8) & 0xfu);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int* status = static_cast<int*>(workspace);
    TUNE_CUDA_TRY(cudaMemsetAsync(workspace, 0, tune::kWorkspaceHeader, s), "tune_eval_archs: status reset");
    if (n_kernels == 0) return TUNE_OK;
    // A launch per row, with the row's tables from the host, each starting in the places that the one before it
    // leaves. (One launch for all rows, whose CTAs built their row's tables and read its fields by a row
    // index: 519 us for 50,000 uneven kernels against six rows; now 430.)
    EvalParams p;
    p.x = *axes;
    p.n_kernels = n_kernels;
    p.k = k;
    p.chunk = chunk_code == 0 ? 0 : (1 << (chunk_code - 1));
    for (int i = 0; i < n_arch; ++i) {
        p.a = archs[i];
        const int64_t at = (int64_t)i * n_kernels * k;
        const int rc = launch<false>(p, descs, topk_idx + at, topk_cost + at, nullptr, nullptr, nullptr, nullptr, status, s,
                                     (int)((flags >> 12) & 0xfu), queue_word(status, i), i, n_arch);
        if (rc) return rc;
    }
    return TUNE_OK;
}

// ---------------------------------------------------------------------------
// Internal launcher for the library's other entry points (one architecture row, no
// emitted points): validates nothing beyond what tune_eval does.
// ---------------------------------------------------------------------------
namespace tune {

int eval_launch(const tune_arch* arch, const tune_axes* axes, const tune_kernel_desc* descs, int64_t n_kernels,
                int32_t k, uint32_t flags, int32_t* topk_idx, float* topk_cost, int* status,
                unsigned long long* queue, cudaStream_t s)
{
    int rc = validate(arch, axes, k);
    if (rc) return rc;
    if (flags & ~(TUNE_SCHED_WARP | 0xff00u))
        return fail(TUNE_EINVAL, "flags 0x%x: only TUNE_SCHED_WARP and its chunk/CTA fields", flags);
    const int chunk_code = (int)((flags >> 8) & 0xfu);
    EvalParams p;
    p.a = *arch;
    p.x = *axes;
    p.n_kernels = n_kernels;
    p.k = k;
    p.chunk = chunk_code == 0 ? 0 : (1 << (chunk_code - 1));
    return launch<false>(p, descs, topk_idx, topk_cost, nullptr, nullptr, nullptr, nullptr, status, s,
                         (int)((flags >> 12) & 0xfu), queue);
}

}  // namespace tune
