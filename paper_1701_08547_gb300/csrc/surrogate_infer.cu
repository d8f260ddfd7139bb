// Surrogate features and ranking: per-point features (tune_features), and
// surrogate_infer — features of every point, ensemble forward, per-point mean
// and spread of the predicted runtime, per-kernel top-k by predicted runtime,
// and a per-kernel fallback to the analytic top-k where the members disagree.
#include <cuda_bf16.h>
#include <stdint.h>
#include <string.h>

#include "features.cuh"
#include "tune_internal.h"

using namespace tune_dev;

namespace {

constexpr int IN = TUNE_SURROGATE_INPUTS;  // feature row width (48 features + zeros)
constexpr int64_t kChunkPoints = 1 << 20;  // points per inference chunk

__device__ __forceinline__ void load_desc(const int4* descs, int64_t kid, Desc& kd)
{
    int4 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = __ldg(descs + kid * 4 + q);
    unpack(v, kd);
}

__device__ __forceinline__ void write_row(__nv_bfloat16* row, const float* f)
{
    __nv_bfloat162* r2 = reinterpret_cast<__nv_bfloat162*>(row);
#pragma unroll
    for (int j = 0; j < kFeatures / 2; ++j) r2[j] = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
    const __nv_bfloat162 z = __floats2bfloat162_rn(0.0f, 0.0f);
#pragma unroll
    for (int j = kFeatures / 2; j < IN / 2; ++j) r2[j] = z;
}

// Features of listed samples (kernel id, canonical point index).
__global__ void features_samples(const __grid_constant__ tune_arch a, const __grid_constant__ tune_axes x,
                                 const int4* __restrict__ descs, const int64_t* __restrict__ skern,
                                 const int32_t* __restrict__ spoint, int64_t n, __nv_bfloat16* out, int* status)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    Desc kd;
    load_desc(descs, skern[i], kd);
    const int size = __popc(kd.tm) * __popc(kd.gm) * __popc(kd.um) * __popc(kd.cm);
    float f[kFeatures];
    if (desc_bad(kd, x) || spoint[i] < 0 || spoint[i] >= size) {
        atomicOr(status, tune::kStatusInvalid);
        for (int j = 0; j < kFeatures; ++j) f[j] = 0.0f;
    } else {
        int tp, gp, up, cp;
        decode_point(kd, spoint[i], tp, gp, up, cp);
        point_features(a, kd, x.t[tp], x.g[gp], x.u[up], x.c[cp], f);
    }
    write_row(out + i * IN, f);
}

// ---- features of every point of a range of kernels ----
//
// A feature depends on the descriptor alone (0-17, 43), on one axis value (18-20 on T; 21
// on G; 22, 24, 25, 39, 40, 44, 46, 47 on U; 23, 28, 42 on C) or on the whole point
// (the 16 others). A warp walks consecutive points, 32 at a time, and keeps the parts of
// the kernel it is in as tables in shared memory, already rounded to BF16: 18 + 32 + 16 +
// 8 + 4 entries computed by one lane each instead of 48 features by every lane. Each part
// is the expression point_features() has for it, so the rows are those of tune_features.
// Rows are staged in shared memory (16-byte units, XOR-swizzled) and leave as fully
// coalesced 16-byte stores; the zero units are staged once, the units with descriptor
// features only when the kernel changes.
//
// Bound: 128 bytes written per point, 20 us per 2^20 points at the copy rate; the integer and
// FP32 work of a point (three logarithms, seven divisions) and the tables come to about as
// much. Measured per 2^20 points of the uneven workload: 45 us, against 202 us for one thread
// per point that evaluated all 48 features, found its axis values with __fns and wrote its
// row 4 bytes at a time. 7 CTAs of 4 warps per SM: 72 registers; a full chunk (2^20 points, 8
// groups a warp) then fills the chip once.
// Tables are built one kernel after the other, about 3 us each by latency, so where 32 points are of more than
// kFeatKernels kernels each lane evaluates its point by itself (feat_point). One member, 16,384 kernels, whole call:
// 1 point each 168 us before the tables, 275 with them alone, 158 now; 4 points 218 / 218 / 190 (eight kernels per
// 32 points; with the line at 8: 221); 8 points 269 / 239 / 240.
struct FeatT {
    float t, lane;  // T; 32 W_B / T
    int wb, gw;
    uint32_t w18;  // features 18, 19
    uint16_t b20, b26;
};
struct FeatG {
    int g;
    uint32_t b21;
};
struct FeatU {
    float cnm, cm;
    int kind, warps, rpw, regs;  // register limit: kind 0: G_R = warps; 1: per warp; 2: per block
    uint32_t w24, w46;           // features 24, 25; 46, 47
    uint16_t b22, b39, b40, b44;
};
struct FeatC {
    int gs;
    uint16_t b23, b28, b42, pad;
};

constexpr int kFeatKernels = 4;  // kernels among 32 points up to which their tables are built (see above)
constexpr int kFeatWarps = 4;
constexpr int kFeatGroups = 8;  // groups of 32 points a warp walks at most (tables are reused along them)

struct alignas(16) FeatWarp {
    uint4 stage[32 * 8];
    FeatT t[32];
    FeatU u[8];
    FeatG g[16];
    FeatC c[4];
    alignas(16) uint16_t d[18];
    uint16_t b43;
    float rcp[7];  // 1 / IPC_c
};

__device__ __forceinline__ uint16_t bf16_bits(float f) { return __bfloat16_as_ushort(__float2bfloat16_rn(f)); }

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    return (uint32_t)bf16_bits(lo) | (uint32_t)bf16_bits(hi) << 16;
}

__device__ __forceinline__ uint32_t join2(uint32_t lo, uint32_t hi) { return (lo & 0xffffu) | hi << 16; }

// Tables of one descriptor, by all lanes of a warp; (vt, vg, vu, vc): the lane's axis values.
__device__ __forceinline__ void feat_tables(const tune_arch& a, const Desc& kd, int lane, int vt, int vg, int vu, int vc,
                                            FeatWarp& s)
{
    const uint32_t below = (1u << lane) - 1u;
    float tot = 0.0f;
#pragma unroll
    for (int c = 0; c < 7; ++c) tot += kd.n[c];
    if (lane < 7) {
        float n = kd.n[0];
#pragma unroll
        for (int c = 1; c < 7; ++c) n = lane == c ? kd.n[c] : n;
        s.d[lane] = bf16_bits(log2f(n + 1.0f) / 20.0f);
        s.d[7 + lane] = bf16_bits(n / (tot + 1.0f));
    } else if (lane == 7) {
        s.d[14] = bf16_bits(
            log2f((kd.n[CL_FP32] + kd.n[CL_FP64] + 1.0f) / (kd.n[CL_GLDST] + kd.n[CL_SLDST] + 1.0f)) / 10.0f);
        s.d[15] = bf16_bits((float)kd.r0 / 255.0f);
        s.d[16] = bf16_bits((float)kd.s0 / 65536.0f);
        s.d[17] = bf16_bits(kd.d);
    }
    if (kd.tm >> lane & 1u) {
        const int T = vt, wb = (T + 31) / 32;
        const int gw = T <= a.max_threads_block ? min(a.max_blocks_sm, a.max_warps_sm / wb) : 0;
        FeatT e;
        e.t = (float)T;
        e.lane = __fdiv_rn((float)(32 * wb), (float)T);
        e.wb = wb;
        e.gw = gw;
        e.w18 = pack2(log2f((float)T) / 10.0f, (float)wb / 32.0f);
        e.b20 = bf16_bits(e.lane);
        e.b26 = bf16_bits((float)min(gw, 64) / 32.0f);
        s.t[__popc(kd.tm & below)] = e;
    }
    if (lane < 16 && (kd.gm >> lane & 1u)) {
        FeatG e;
        e.g = vg;
        e.b21 = bf16_bits(log2f((float)vg) / 16.0f);
        s.g[__popc(kd.gm & below)] = e;
    }
    if (lane < 8 && (kd.um >> lane & 1u)) {
        const int U = vu, R = kd.r0 + 4 * (U - 1);
        FeatU e;
        e.kind = 0;
        e.warps = 0;
        e.rpw = 0;
        e.regs = R;
        if (R > a.regs_thread_max) {
            e.warps = 0;
        } else if (R <= 0) {
            e.warps = a.max_blocks_sm;
        } else if (a.reg_alloc_mode == 0) {
            e.kind = 1;
            e.rpw = ceil_div(R * 32, a.reg_alloc_unit) * a.reg_alloc_unit;
            e.warps = (a.regs_sm / e.rpw) / a.warp_alloc_gran * a.warp_alloc_gran;
        } else {
            e.kind = 2;
        }
        unit_costs(kd.n, kd.d, U, s.rcp, a.work_scale, e.cnm, e.cm);
        const float f39 = log2f(e.cnm + 1.0f) / 40.0f, f40 = log2f(e.cm + 1.0f) / 40.0f;
        e.w24 = pack2((float)R / 255.0f, (float)e.rpw / 8192.0f);
        e.w46 = pack2((f39 - __bfloat162float(__float2bfloat16_rn(f39))) * 256.0f,
                      (f40 - __bfloat162float(__float2bfloat16_rn(f40))) * 256.0f);
        e.b22 = bf16_bits((float)U / 8.0f);
        e.b39 = bf16_bits(f39);
        e.b40 = bf16_bits(f40);
        e.b44 = bf16_bits(log2f(__fdiv_rn(kd.n[CL_BRANCH], (float)U) + 1.0f) / 20.0f);
        s.u[__popc(kd.um & below)] = e;
    }
    int s_alloc = 0;
    if (kd.s0 <= a.smem_block_max)
        s_alloc = ceil_div(kd.s0 + a.smem_reserved_block, a.smem_alloc_unit) * a.smem_alloc_unit;
    if (lane < 4 && (kd.cm >> lane & 1u)) {
        const int C = vc, gs = smem_blocks(a, kd.s0, C);
        int cap = 0;
        if (kd.s0 <= a.smem_block_max) {
            const int max_cap = a.smem_caps[a.n_smem_caps - 1];
            for (int i = 0; i < a.n_smem_caps; ++i) {
                const int ci = a.smem_caps[i];
                if (100LL * ci >= (long long)C * max_cap && ci >= s_alloc) {
                    cap = ci;
                    break;
                }
            }
        }
        FeatC e;
        e.gs = gs;
        e.b23 = bf16_bits((float)C / 100.0f);
        e.b28 = bf16_bits((float)min(gs, 64) / 32.0f);
        e.b42 = bf16_bits((float)cap / 233472.0f);
        s.c[__popc(kd.cm & below)] = e;
    }
    if (lane == 8) s.b43 = bf16_bits((float)s_alloc / 65536.0f);
}

// The row of point p of descriptor kid by one lane, staged like the others; returns its validity.
__device__ __forceinline__ bool feat_point(const tune_arch& a, const tune_axes& x, const int4* descs, int64_t kid, int64_t p,
                                           uint4* row, int sx, int* status)
{
    Desc kd;
    load_desc(descs, kid, kd);
    const int size = __popc(kd.tm) * __popc(kd.gm) * __popc(kd.um) * __popc(kd.cm);
    if (desc_bad(kd, x) || p >= size) {
        atomicOr(status, tune::kStatusInvalid);
#pragma unroll
        for (int j = 0; j < kFeatures / 8; ++j) row[j ^ sx] = make_uint4(0, 0, 0, 0);
        return false;
    }
    int tp, gp, up, cp;
    decode_point(kd, (int)p, tp, gp, up, cp);
    float f[kFeatures];
    point_features(a, kd, x.t[tp], x.g[gp], x.u[up], x.c[cp], f);
#pragma unroll
    for (int j = 0; j < kFeatures / 8; ++j)
        row[j ^ sx] = make_uint4(pack2(f[8 * j], f[8 * j + 1]), pack2(f[8 * j + 2], f[8 * j + 3]),
                                 pack2(f[8 * j + 4], f[8 * j + 5]), pack2(f[8 * j + 6], f[8 * j + 7]));
    return f[29] > 0.0f;  // B* > 0
}

// Row i of the chunk = global point p0 + i (p0 = pt_off[k0]) of kernels [k0, k1); a point's
// kernel is found by a binary search over the offsets (the chunk's few offsets stay in L1).
// Also writes score[i] = 0 where the point is valid (B* > 0), +inf elsewhere.
__global__ void __launch_bounds__(32 * kFeatWarps, 7)
    features_points(const __grid_constant__ tune_arch a, const __grid_constant__ tune_axes x,
                    const int4* __restrict__ descs, const int64_t* __restrict__ pt_off, int64_t k0, int64_t k1,
                    int64_t p0, int64_t np, int groups, __nv_bfloat16* out, float* score, int* status)
{
    __shared__ FeatWarp sw[kFeatWarps];
    const int lane = threadIdx.x & 31;
    FeatWarp& s = sw[threadIdx.x >> 5];
    const int64_t beg = ((int64_t)blockIdx.x * kFeatWarps + (threadIdx.x >> 5)) * groups * 32;
    if (beg >= np) return;
    const int64_t end = beg + groups * 32 < np ? beg + groups * 32 : np;
    const int vt = x.t[lane], vg = lane < 16 ? x.g[lane] : 1, vu = lane < 8 ? x.u[lane] : 1;
    const int vc = lane < 4 ? x.c[lane] : 0;
    if (lane < 7) s.rcp[lane] = __fdiv_rn(1.0f, a.ipc[lane]);
    const uint4 zero = make_uint4(0, 0, 0, 0);
    uint4* row = s.stage + lane * 8;  // the lane's staged row; unit j is at j ^ (lane & 7)
    const int sx = lane & 7;
    row[6 ^ sx] = zero;
    row[7 ^ sx] = zero;

    // rows start at 16-byte boundaries unless the caller's workspace does not
    const bool aligned = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    int64_t cur = -1, cur_beg = 0, cur_end = 0;  // the kernel of the tables and its points
    bool cur_bad = false, staged = false;        // staged: every row's units 0, 1 are cur's
    int size = 0, nC = 1, nU = 1, nG = 1;
    float rC = 1.0f, rU = 1.0f, rG = 1.0f;

    for (int64_t base = beg; base < end; base += 32) {
        const int64_t gp = p0 + base + lane;
        const bool on = base + lane < end;
        int64_t lo = cur;
        if (__any_sync(0xffffffffu, on && (cur < 0 || gp < cur_beg || gp >= cur_end))) {
            lo = k0;
            int64_t hi = k1;  // pt_off[lo] <= gp < pt_off[hi]
            while (hi - lo > 1) {
                const int64_t mid = (lo + hi) >> 1;
                if (pt_off[mid] <= gp)
                    lo = mid;
                else
                    hi = mid;
            }
        }
        bool valid = false;
        unsigned todo = __ballot_sync(0xffffffffu, on);
        const int64_t left = __shfl_up_sync(0xffffffffu, lo, 1);
        const unsigned firsts = __ballot_sync(0xffffffffu, on && (lane == 0 || lo != left));
        if (__popc(firsts) > kFeatKernels) {
            if (on) valid = feat_point(a, x, descs, lo, gp - pt_off[lo], row, sx, status);
            staged = false;
            todo = 0;
        }
        while (todo) {
            const int64_t kid = __shfl_sync(0xffffffffu, lo, __ffs(todo) - 1);
            const unsigned mine = __ballot_sync(0xffffffffu, on && lo == kid);
            todo &= ~mine;
            if (kid != cur) {
                int4 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = __ldg(descs + kid * 4 + q);
                Desc kd;
                unpack(v, kd);
                cur = kid;
                cur_beg = pt_off[kid];
                cur_end = pt_off[kid + 1];
                cur_bad = desc_bad(kd, x);
                staged = false;
                nC = __popc(kd.cm);
                nU = __popc(kd.um);
                nG = __popc(kd.gm);
                size = __popc(kd.tm) * nG * nU * nC;
                rC = __fdiv_rn(1.0f, (float)nC);
                rU = __fdiv_rn(1.0f, (float)nU);
                rG = __fdiv_rn(1.0f, (float)nG);
                __syncwarp();  // the previous tables have been read
                if (!cur_bad) feat_tables(a, kd, lane, vt, vg, vu, vc, s);
                __syncwarp();
            }
            const int64_t p64 = gp - cur_beg;
            if (on && lo == kid) {
                if (cur_bad || p64 >= size) {
                    atomicOr(status, tune::kStatusInvalid);
#pragma unroll
                    for (int j = 0; j < 6; ++j) row[j ^ sx] = zero;
                } else {
                    // axis positions; p < 2^14 and each divisor <= 16: (p + 1/2) / d is at least
                    // 1/32 away from a whole number, far more than the two roundings move it
                    int p = (int)p64;
                    int q = (int)(((float)p + 0.5f) * rC);
                    const FeatC& ec = s.c[p - q * nC];
                    p = q;
                    q = (int)(((float)p + 0.5f) * rU);
                    const FeatU& eu = s.u[p - q * nU];
                    p = q;
                    q = (int)(((float)p + 0.5f) * rG);
                    const FeatG& eg = s.g[p - q * nG];
                    const FeatT& et = s.t[q];

                    const int wb = et.wb, G = eg.g, gw = et.gw, gs = ec.gs;
                    int gr;
                    if (eu.kind == 0) {
                        gr = eu.warps;
                    } else if (eu.kind == 1) {
                        gr = eu.rpw * wb > a.regs_block_max ? 0 : eu.warps / wb;
                    } else {
                        const long long rpb =
                            (long long)ceil_div(eu.regs * 32 * wb, a.reg_alloc_unit) * a.reg_alloc_unit;
                        gr = rpb > a.regs_block_max ? 0 : (int)(a.regs_sm / rpb);
                    }
                    const int B = min(gw, min(gr, gs));
                    const int W = B * wb;
                    valid = B > 0;
                    float waves = 0.0f, par = 0.0f, hide = 0.0f, cost = 0.0f;
                    if (B > 0) {
                        const int slots = a.n_sm * B;
                        const int wv = ceil_div(G, slots);
                        waves = (float)wv;
                        par = __fdiv_rn((float)(a.n_sm * G), (float)(wv * slots));
                        hide = fmaxf(1.0f, __fdiv_rn((float)a.w_sat, (float)W));
                        const float X = __fmul_rn(__fmaf_rn(eu.cm, hide, eu.cnm), et.lane);
                        cost = __fmul_rn(X, __fdiv_rn((float)(wv * slots), (float)(a.n_sm * G)));
                    }
                    const float f38 = log2f(cost + 1.0f) / 40.0f;
                    const uint32_t one = 0x3f80;  // BF16 1.0
                    const uint32_t b32 = valid && gw == B ? one : 0, b33 = valid && gr == B ? one : 0;
                    const uint32_t b34 = valid && gs == B ? one : 0;
                    if (!staged) {
                        row[0 ^ sx] = *reinterpret_cast<const uint4*>(s.d);
                        row[1 ^ sx] = *reinterpret_cast<const uint4*>(s.d + 8);
                    }
                    row[2 ^ sx] = make_uint4(*reinterpret_cast<const uint32_t*>(s.d + 16), et.w18,
                                             join2(et.b20, eg.b21), join2(eu.b22, ec.b23));
                    row[3 ^ sx] = make_uint4(eu.w24, join2(et.b26, bf16_bits((float)min(gr, 64) / 32.0f)),
                                             join2(ec.b28, bf16_bits((float)B / 32.0f)),
                                             pack2((float)W / 64.0f, (float)W / (float)a.max_warps_sm));
                    row[4 ^ sx] = make_uint4(join2(b32, b33),
                                             join2(b34, bf16_bits(waves > 0.0f ? log2f(waves) / 10.0f : 0.0f)),
                                             pack2(par / (float)a.n_sm, hide / 32.0f),
                                             join2(bf16_bits(f38), eu.b39));
                    row[5 ^ sx] = make_uint4(
                        join2(eu.b40, bf16_bits(log2f((float)G * et.t) / 26.0f)), join2(ec.b42, s.b43),
                        join2(eu.b44, bf16_bits((f38 - __bfloat162float(__float2bfloat16_rn(f38))) * 256.0f)),
                        eu.w46);
                }
            }
            staged = mine == 0xffffffffu && !__any_sync(0xffffffffu, cur_bad || p64 >= size);
        }
        __syncwarp();
        if (on) score[base + lane] = valid ? 0.0f : __int_as_float(0x7f800000);
        const int rows = (int)(end - base < 32 ? end - base : 32);
        if (aligned) {
            uint4* dst = reinterpret_cast<uint4*>(out + base * IN);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = i * 4 + (lane >> 3), j = lane & 7;
                if (r < rows) dst[i * 32 + lane] = s.stage[r * 8 + (j ^ (r & 7))];
            }
        } else {  // a word of a row per lane
            const uint32_t* src = reinterpret_cast<const uint32_t*>(s.stage);
            uint32_t* dst = reinterpret_cast<uint32_t*>(out + base * IN);
            for (int r = 0; r < rows; ++r) dst[r * 32 + lane] = src[(r * 8 + ((lane >> 2) ^ (r & 7))) * 4 + (lane & 3)];
        }
        __syncwarp();  // the staged rows have been read
    }
}

// Chunk-relative segment offsets: rel[j] = pt_off[k0 + j] - pt_off[k0], j = 0..nk.
__global__ void rebase_offsets(const int64_t* __restrict__ pt_off, int64_t k0, int64_t nk, int64_t* rel)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j <= nk) rel[j] = pt_off[k0 + j] - pt_off[k0];
}

// Per point: runtime estimate = mean over members of exp(prediction); spread = std / mean;
// invalid points (score[i] = +inf from features_points) keep +inf. Bound by reading members * 4
// bytes a point: 9.8 us per 2^20 points (26 us when it read validity from the feature rows, one
// 32-byte sector per point).
__global__ void score_points(const float* __restrict__ pred, int64_t n, int members, float* score, float* spread)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const bool valid = score[i] == 0.0f;
    float s = 0.0f, s2 = 0.0f;
    for (int m = 0; m < members; ++m) {
        const float r = expf(pred[(int64_t)m * n + i]);
        s += r;
        s2 += r * r;
    }
    const float mean = s / members;
    const float var = fmaxf(s2 / members - mean * mean, 0.0f);
    score[i] = valid ? mean : __int_as_float(0x7f800000);
    spread[i] = valid ? sqrtf(var) / mean : 0.0f;
}

// Per kernel: use the analytic top-k if any of the surrogate's top-k points has spread > thresh.
__global__ void apply_fallback(const int32_t* __restrict__ s_idx, const float* __restrict__ s_val,
                               const int32_t* __restrict__ a_idx, const float* __restrict__ a_val,
                               const float* __restrict__ spread, const int64_t* __restrict__ pt_off, int64_t k0,
                               int64_t nk, int k, float thresh, int32_t* out_idx, float* out_val, uint8_t* flag)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nk) return;
    const int64_t kid = k0 + j;
    const int64_t base = pt_off[kid] - pt_off[k0];
    bool fb = false;
    for (int r = 0; r < k; ++r) {
        const int p = s_idx[j * k + r];
        if (p >= 0 && spread[base + p] > thresh) fb = true;
    }
    flag[kid] = fb ? 1 : 0;
    for (int r = 0; r < k; ++r) {
        out_idx[kid * k + r] = fb ? a_idx[kid * k + r] : s_idx[j * k + r];
        out_val[kid * k + r] = fb ? a_val[kid * k + r] : s_val[j * k + r];
    }
}

int64_t align256(int64_t b) { return (b + 255) & ~int64_t(255); }

}  // namespace

extern "C" {

int tune_features(const tune_arch* arch, const tune_axes* axes, const tune_kernel_desc* descs,
                  const int64_t* sample_kernel, const int32_t* sample_point, int64_t n, uint16_t* feats,
                  void* workspace, size_t ws_bytes, tune_stream_t stream)
{
    tune::clear_error();
    if (!arch || !axes || !workspace || ws_bytes < tune::kWorkspaceHeader || n < 0)
        return tune::fail(TUNE_EINVAL, "tune_features: bad arguments");
    if (n > 0 && (!descs || !sample_kernel || !sample_point || !feats))
        return tune::fail(TUNE_EINVAL, "tune_features: NULL array");
    int rc = tune::validate_inputs(arch, axes);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    TUNE_CUDA_TRY(cudaMemsetAsync(workspace, 0, tune::kWorkspaceHeader, s), "tune_features: status reset");
    if (n == 0) return TUNE_OK;
    features_samples<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(
        *arch, *axes, reinterpret_cast<const int4*>(descs), sample_kernel, sample_point, n,
        reinterpret_cast<__nv_bfloat16*>(feats), static_cast<int*>(workspace));
    TUNE_CUDA_TRY(cudaGetLastError(), "tune_features: launch");
    return TUNE_OK;
}

}  // extern "C"

// surrogate_infer needs the handle's forward; declared in surrogate.cu.
extern "C" int surrogate_forward(tune_surrogate* h, const uint16_t* feats, int64_t n, float* pred,
                                 tune_stream_t stream);
extern "C" int surrogate_members(const tune_surrogate* h);

extern "C" size_t surrogate_infer_workspace_bytes(int members, int64_t n_kernels, int32_t k)
{
    int64_t b = 2 * tune::kWorkspaceHeader;           // status; header for the internal calls
    b += align256(kChunkPoints * IN * 2);              // features
    b += align256((int64_t)members * kChunkPoints * 4); // predictions
    b += 2 * align256(kChunkPoints * 4);                // score, spread
    b += align256((int64_t)(kChunkPoints / 64 + 2) * 8);  // chunk offsets (>= 64 points per kernel? sized below)
    b += 2 * align256(n_kernels * k * 4);               // analytic top-k
    b += 2 * align256(n_kernels * k * 4);               // surrogate top-k (per chunk, sized for all)
    b += align256((n_kernels + 1) * 8);                 // device offsets
    return (size_t)b;
}

extern "C" int surrogate_infer(tune_surrogate* h, const tune_arch* arch, const tune_axes* axes,
                               const tune_kernel_desc* descs, int64_t n_kernels, const int64_t* pt_offsets_host,
                               int32_t k, float thresh, int32_t* topk_idx, float* topk_score,
                               uint8_t* used_fallback, void* workspace, size_t ws_bytes, tune_stream_t stream)
{
    tune::clear_error();
    if (!h || !arch || !axes || !pt_offsets_host || k < 1 || k > 16 || n_kernels < 0)
        return tune::fail(TUNE_EINVAL, "surrogate_infer: bad arguments");
    const int members = surrogate_members(h);
    if (!workspace || ws_bytes < surrogate_infer_workspace_bytes(members, n_kernels, k))
        return tune::fail(TUNE_ENOMEM, "surrogate_infer: workspace smaller than surrogate_infer_workspace_bytes()");
    if (n_kernels == 0) return TUNE_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    char* w = static_cast<char*>(workspace);
    int* status = reinterpret_cast<int*>(w);
    w += tune::kWorkspaceHeader;
    void* inner = w;  // workspace header of the tune_eval / tune_topk calls made here
    w += tune::kWorkspaceHeader;
    auto* feats = reinterpret_cast<__nv_bfloat16*>(w);
    w += align256(kChunkPoints * IN * 2);
    float* pred = reinterpret_cast<float*>(w);
    w += align256((int64_t)members * kChunkPoints * 4);
    float* score = reinterpret_cast<float*>(w);
    w += align256(kChunkPoints * 4);
    float* spread = reinterpret_cast<float*>(w);
    w += align256(kChunkPoints * 4);
    int64_t* coff = reinterpret_cast<int64_t*>(w);  // chunk-relative offsets, reused per chunk
    w += align256((int64_t)(kChunkPoints / 64 + 2) * 8);
    int32_t* a_idx = reinterpret_cast<int32_t*>(w);
    w += align256(n_kernels * k * 4);
    float* a_val = reinterpret_cast<float*>(w);
    w += align256(n_kernels * k * 4);
    int32_t* s_idx = reinterpret_cast<int32_t*>(w);
    w += align256(n_kernels * k * 4);
    float* s_val = reinterpret_cast<float*>(w);
    w += align256(n_kernels * k * 4);
    int64_t* d_off = reinterpret_cast<int64_t*>(w);

    const int64_t sms = tune::device_sm_count();
    if (sms <= 0) return tune::fail(TUNE_ECUDA, "surrogate_infer: cannot query the SM count");
    TUNE_CUDA_TRY(cudaMemsetAsync(status, 0, tune::kWorkspaceHeader, s), "surrogate_infer: status reset");
    // Analytic top-k of every kernel (the fallback).
    int rc = tune_eval(arch, axes, descs, n_kernels, k, TUNE_SCHED_WARP, a_idx, a_val, nullptr, nullptr, nullptr,
                       nullptr, inner, tune::kWorkspaceHeader, stream);
    if (rc) return rc;
    TUNE_CUDA_TRY(cudaMemcpyAsync(d_off, pt_offsets_host, (n_kernels + 1) * 8, cudaMemcpyHostToDevice, s),
                  "surrogate_infer: offsets");
    int64_t k0 = 0;
    while (k0 < n_kernels) {
        // Chunk: as many whole kernels as fit kChunkPoints (and the offsets scratch).
        int64_t k1 = k0;
        while (k1 < n_kernels && pt_offsets_host[k1 + 1] - pt_offsets_host[k0] <= kChunkPoints &&
               k1 - k0 < kChunkPoints / 64)
            ++k1;
        if (k1 == k0) return tune::fail(TUNE_EINVAL, "surrogate_infer: a space larger than the chunk");
        const int64_t np = pt_offsets_host[k1] - pt_offsets_host[k0];
        const int64_t nk = k1 - k0;
        // Everything below is stream-ordered: the chunk buffers are reused without a host wait.
        rebase_offsets<<<(unsigned)((nk + 1 + 255) / 256), 256, 0, s>>>(d_off, k0, nk, coff);
        TUNE_CUDA_TRY(cudaGetLastError(), "surrogate_infer: offsets launch");
        if (np > 0) {
            // a warp's walk: long where every SM still gets 16 warps, so that few points stay parallel
            const int64_t want = np / (32 * 16 * sms);
            const int groups = (int)(want < 1 ? 1 : want > kFeatGroups ? kFeatGroups : want);
            const int64_t per_cta = (int64_t)groups * 32 * kFeatWarps;
            features_points<<<(unsigned)((np + per_cta - 1) / per_cta), 32 * kFeatWarps, 0, s>>>(
                *arch, *axes, reinterpret_cast<const int4*>(descs), d_off, k0, k1, pt_offsets_host[k0], np, groups,
                feats, score, status);
            TUNE_CUDA_TRY(cudaGetLastError(), "surrogate_infer: features launch");
            rc = surrogate_forward(h, reinterpret_cast<const uint16_t*>(feats), np, pred, stream);
            if (rc) return rc;
            score_points<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(pred, np, members, score, spread);
            TUNE_CUDA_TRY(cudaGetLastError(), "surrogate_infer: score launch");
        }
        rc = tune_topk(score, coff, nk, k, s_idx, s_val, inner, tune::kWorkspaceHeader, stream);
        if (rc) return rc;
        apply_fallback<<<(unsigned)((nk + 127) / 128), 128, 0, s>>>(s_idx, s_val, a_idx, a_val, spread, d_off, k0, nk,
                                                                   k, thresh, topk_idx, topk_score, used_fallback);
        TUNE_CUDA_TRY(cudaGetLastError(), "surrogate_infer: fallback launch");
        k0 = k1;
    }
    int st = 0;
    TUNE_CUDA_TRY(cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, s), "surrogate_infer: status");
    TUNE_CUDA_TRY(cudaStreamSynchronize(s), "surrogate_infer: sync");
    if (st) return tune::fail(TUNE_EINVAL, "surrogate_infer: a descriptor was malformed");
    return TUNE_OK;
}
